// Shrink for small decode batches: z[t] = s_a * A_a x[t] for tokens scattered across adapters
// (paper Section 2.1 for A: r x h_in; Section 4.3: tokens that share an adapter are handled as one
// sub-batch so the adapter is fetched once), with the routing derived inside the kernel so that a
// step of a few microseconds needs no routing launch.  Larger batches take the tensor-core tiles of
// shrink_tiles.cu.
#include "decode_route.cuh"
#include "internal.cuh"
#include "launch.cuh"
#include "ptx.cuh"
#include "shrink_rows.cuh"

namespace edgelora {

// ---------------------------------------------------------------------------------------------
// Decode shrink with the routing folded in (batches of at most 256 tokens).
//
// A decode step is a few microseconds long, so a separate routing launch would cost as much as
// the arithmetic.  Here every CTA derives the u-batches (paper Section 3.4) from the ids itself, in
// shared memory, and then takes its share of the work items (group, K chunk).  An item streams the
// live rows of A_a over its K chunk once from HBM with TMA copies into a private shared-memory
// ring (three K steps of eight rows ahead per warp), and dots them with the x rows of
// up to four tokens of the group at a time (a group's tokens are cut into blocks of eight, each
// block an item of its own, so that a popular adapter does not serialise on one CTA); lanes are
// reduced by shuffles.  Items belong to single warps, which run independently so that the fixed
// latencies of one overlap the streaming of the others.  Partial sums go to
// zws[chunk][token][row]; whichever warp finishes a (group, eight rows) last adds the chunks in a
// fixed order into the final plane zws[kMaxZSplits] that the base-product kernel reads.  The last CTA also
// writes the routing plan in its canonical form for the base-product kernel and for export.

constexpr int kDsTicket = kDecodeMaxT * 8;  // index of the work-item ticket counter in group_counters

constexpr size_t ds_ring_bytes(int depth) {
  return static_cast<size_t>(kShrinkThreads / 32) * depth * kDsStageBytes + 1024;
}

// kDsDepth = 4 fills an SM's shared memory (large batches: bandwidth); kDsDepth = 2 leaves room
// for a CTA of the base-product kernel beside it (small batches: the two kernels overlap).
template <int kDsDepth, bool kQ8>
__global__ void __launch_bounds__(kShrinkThreads, 2)  // <= 128 registers: fits beside the base-product CTAs
decode_shrink_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_d,
                     const __grid_constant__ CUtensorMap tmap_x,
                     const int32_t *__restrict__ ids, const SlotRow *__restrict__ slots,
                     PlanView pv, float *__restrict__ zws, int32_t *__restrict__ group_counters,
                     int32_t T, int32_t h_in, int32_t R_pad, int32_t n_slots, int32_t max_tokens,
                     int32_t target_items, int32_t fill_warps, int32_t late_ticket, uint32_t *status) {
  extern __shared__ uint8_t s_ring_raw[];  // [warp][stage][8 A rows + 4 x rows][512 bytes]
  __shared__ uint64_t s_bars[kShrinkThreads / 32][kDsMaxDepth];
  __shared__ Groups s_groups;
  __shared__ int32_t s_grank[256];     // rank and scale of each group's slot
  __shared__ float s_gscale[256];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  ptx::pdl_launch_dependents();
  if (tid == 0) {
    ptx::prefetch_tensormap(&tmap_a);
    ptx::prefetch_tensormap(&tmap_x);
  }
  if (lane < kDsMaxDepth) {  // every warp sets up its own ring barriers
    ptx::mbar_init(&s_bars[warp][lane], 1);
    ptx::fence_barrier_init();
  }

  // ---- routing, in shared memory (reads only the caller's ids)
  const bool bad = derive_groups<kDsTok, 1, kShrinkThreads>(s_groups, ids, T, n_slots, tid);
  const int G = s_groups.n_groups, NB = s_groups.n_blocks;
  if (tid < G) {
    const SlotRow row = slots[s_groups.adapter[tid]];
    s_grank[tid] = row.rank;
    s_gscale[tid] = row.scale;
  }
  const int any_bad = __syncthreads_or(bad ? 1 : 0);

  // Work items are per warp: (token block, K chunk, group of eight rank rows).  K chunks: enough
  // items for every warp of the grid, but a chunk keeps at least four K steps (1024 elements)
  // unless h_in is shorter, so that the ring's ramp-up is amortised; or two, as long as a warp has no more than one item
  // (fill_warps: so many of them, none where the caller gave the number of items).
  const int n_ksteps = (h_in + 255) >> 8, warps_total = (gridDim.x - 1) * (kShrinkThreads / 32);
  const int n_rgn = R_pad >> 3;  // row groups of the rank stride: 2, 4 or 8
  int KS = (target_items + max(NB * n_rgn, 1) - 1) / max(NB * n_rgn, 1);
  KS = max(1, min(min(KS, kMaxZSplits), n_ksteps / 4));
  if (NB * n_rgn * KS < fill_warps)
    KS = max(KS, min(min(kMaxZSplits, n_ksteps / 2), fill_warps / max(NB * n_rgn, 1)));
  const int spc = (n_ksteps + KS - 1) / KS;
  KS = (n_ksteps + spc - 1) / spc;

  // Earlier kernels on the stream may still read the plan and z, so every write to them below comes
  // after griddepcontrol.wait; the operand loads (the pool and x are not written by this library's
  // kernels) start before it.
  const bool publisher = blockIdx.x == gridDim.x - 1;

  // ---- the last CTA publishes the plan in canonical order (ids ascending, -1 first): everything
  // is worked out in shared memory and registers first, the stores come after the wait
  if (publisher) publish_decode_plan(pv, s_groups.id[tid], T, any_bad, KS, s_groups.id, s_groups.cnt, s_groups.wt);

  // ---- per-warp work items, no CTA-wide synchronisation from here on
  const int n_items = NB * KS * n_rgn;
  const size_t zplane = static_cast<size_t>(max_tokens) * R_pad;
  uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(s_ring_raw) + 127) & ~uintptr_t(127)) +
                  static_cast<size_t>(warp) * kDsDepth * kDsStageBytes;
  uint64_t *bars = s_bars[warp];
  uint32_t phase = 0;
  bool ok = true, waited = publisher;
  // Items are drawn from a ticket counter so that warps stay busy whatever the items cost; the
  // next ticket is drawn before the current item is processed.  The very last draw of the launch
  // (item number n_items + warps - 1) puts the counter back to zero.
  // (the publishing CTA takes no items: nothing that the next kernel waits for queues behind it)
  int32_t *ticket = group_counters + kDsTicket;
  int item = publisher ? n_items : blockIdx.x * (kShrinkThreads / 32) + warp;  // first round is static
  // The warp that completes a (group, row group) adds the K chunks in order into the final plane;
  // it never waits for the others.  (Run at the end of the item, with the ring drained: its
  // release is a fence, and a fence behind copies in flight waits for them too - putting it off
  // into the next item's ramp-up measured slower.)
  int pend_gi = -1, pend_rg = 0, pend_gt0 = 0, pend_gend = 0;
  auto finalize = [&]() {
    if (pend_gi < 0) return;
    const int arrivals = KS * ((pend_gend - pend_gt0 + kDsTok - 1) / kDsTok);
    __syncwarp();  // the lanes' z stores happen before lane 0's release
    int old = 0;
    if (lane == 0) old = atomic_add_acq_rel(&group_counters[pend_gi * 8 + pend_rg], 1);
    old = __shfl_sync(0xffffffffu, old, 0);
    if (old == arrivals - 1) {
      if (lane == 0) group_counters[pend_gi * 8 + pend_rg] = 0;  // ready for the next launch
      add_z_planes(zws, zplane, KS, s_groups.tok + pend_gt0, pend_gend - pend_gt0, R_pad, pend_rg * 8, lane);
    }
    pend_gi = -1;
  };
  // When this launch may start under the kernels of the call before it (late_ticket), another
  // instance of this kernel can still be running, and the counter is theirs until this warp's
  // dependency wait has returned: the draw then comes after the wait, at the end of the item.
  const bool use_tickets = n_items > warps_total;  // otherwise the static first round is everything
  auto draw = [&]() {
    if (!use_tickets) return n_items;
    if (!waited) {
      ptx::pdl_wait_prior_grids();
      waited = true;
    }
    int n = 0;
    if (lane == 0) n = warps_total + atomicAdd(ticket, 1);
    return __shfl_sync(0xffffffffu, n, 0);
  };
  while (ok && item < n_items) {
    int next = 0;
    if (!late_ticket) {
      if (lane == 0 && use_tickets) next = warps_total + atomicAdd(ticket, 1);
      next = use_tickets ? __shfl_sync(0xffffffffu, next, 0) : n_items;
    }
    const int cur = item;
    // consecutive items are the K chunks of one (token block, row group), and chunk c takes the K
    // steps c, c + KS, c + 2 KS, ...: warps that run side by side fetch neighbouring 512-byte
    // pieces of the same rows at about the same time
    const int c = cur % KS;
    const int br = cur / KS;
    const int bi = br / n_rgn, rg = br - bi * n_rgn;
    const int gi = s_groups.block_group[bi];
    const int ad = s_groups.adapter[gi];
    const int rank = s_grank[gi];
    const float scale = s_gscale[gi];
    const int gt0 = s_groups.start[gi], g_end = s_groups.start[gi + 1];
    const int t0 = s_groups.block_pos[bi], t1 = min(t0 + kDsTok, g_end);
    if (rank <= 0) {
      if (lane == 0 && c == 0 && rg == 0 && t0 == gt0) atomicOr(status, EDGELORA_STATUS_SLOT_EMPTY);
      item = late_ticket ? draw() : next;
      continue;
    }
    const int n_rg = (rank + 7) >> 3;  // live groups of eight rows
    if (rg >= n_rg) {  // rows past the rank are zero padding: nothing to do
      item = late_ticket ? draw() : next;
      continue;
    }
    const int step0 = c, step1 = n_ksteps;
    const int q = lane & 3, r = rg * 8 + (lane >> 2);
    for (int tb = t0; ok && tb < t1; tb += kDsTok) {
      const int nt = min(kDsTok, t1 - tb);
      float acc[8 * kDsTok];
#pragma unroll
      for (int i = 0; i < 8 * kDsTok; ++i) acc[i] = 0.f;
      int32_t tok[kDsTok];
#pragma unroll
      for (int qq = 0; qq < kDsTok; ++qq) tok[qq] = s_groups.tok[tb + min(qq, nt - 1)];
      if (nt == 1) ok = shrink_rows8<1, kDsDepth, kQ8>(&tmap_a, &tmap_d, &tmap_x, ad, rg * 8, tok, step0, step1, KS, ring, bars, phase, lane, acc);
      else if (nt == 2) ok = shrink_rows8<2, kDsDepth, kQ8>(&tmap_a, &tmap_d, &tmap_x, ad, rg * 8, tok, step0, step1, KS, ring, bars, phase, lane, acc);
      else if (nt == 3) ok = shrink_rows8<3, kDsDepth, kQ8>(&tmap_a, &tmap_d, &tmap_x, ad, rg * 8, tok, step0, step1, KS, ring, bars, phase, lane, acc);
      else ok = shrink_rows8<4, kDsDepth, kQ8>(&tmap_a, &tmap_d, &tmap_x, ad, rg * 8, tok, step0, step1, KS, ring, bars, phase, lane, acc);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      sum_over_lanes(acc, lane);  // value L: row L / 4, token L % 4
      if (!waited) {  // first write of this warp to memory that earlier kernels may read
        ptx::pdl_wait_prior_grids();
        waited = true;
      }
      if (q < nt && EL_CHECK(status, s_groups.tok[tb + q] < max_tokens && ad >= 0 && ad < n_slots, 20))
        zws[(KS > 1 ? c : kMaxZSplits) * zplane + static_cast<size_t>(s_groups.tok[tb + q]) * R_pad + r] =
            scale * acc[0];
    }
    if (!ok) break;
    item = late_ticket ? draw() : next;
    if (KS > 1) {
      pend_gi = gi;
      pend_rg = rg;
      pend_gt0 = gt0;
      pend_gend = g_end;
      finalize();
    }
  }
  // Every warp stops at its first ticket >= n_items, so exactly n_items - (first round) + warps
  // draws happen; the one that drew the last ticket resets the counter for the next launch.
  if (lane == 0 && ok && !publisher && use_tickets) {
    const int first_round = min(n_items, warps_total);
    const int last_ticket = warps_total + (n_items - first_round) + first_round - 1;
    if (item == last_ticket) *ticket = 0;
  }
  if (!ok) {
    if (lane == 0) atomicOr(status, EDGELORA_STATUS_TIMEOUT);
    ptx::settle_inline();
  }
}

// The shared-memory limit is an attribute of (function, device): set for the current device, by
// edgelora_pool_create, so that every device a pool lives on is configured.
cudaError_t shrink_set_smem_limit() {
  cudaError_t e = cudaSuccess;
  const int b4 = static_cast<int>(ds_ring_bytes(4)), b2 = static_cast<int>(ds_ring_bytes(2));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(decode_shrink_kernel<4, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, b4);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(decode_shrink_kernel<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, b2);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(decode_shrink_kernel<4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, b4);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(decode_shrink_kernel<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, b2);
  return e;
}

cudaError_t launch_decode_shrink(const CUtensorMap &tmap_a, const CUtensorMap &tmap_d, const CUtensorMap &tmap_x,
                                 const int32_t *ids, const SlotRow *slots, const PlanView &pv,
                                 float *zws, int32_t *group_counters, int32_t T, int32_t h_in,
                                 int32_t R_pad, int32_t n_slots, int32_t max_tokens,
                                 int32_t target_items, int32_t fill_warps, int32_t grid, uint32_t *status, bool pdl, bool a_q8,
                                 int32_t depth, cudaStream_t stream) {
  const int32_t late_ticket = pdl ? 1 : 0;  // pdl here = this launch may start under the call before it
#define EDGELORA_SHRINK(D, Q)                                                                                     \
  launch_ex(decode_shrink_kernel<D, Q>, dim3(grid), dim3(kShrinkThreads), ds_ring_bytes(D), stream, pdl, 1, tmap_a, \
            tmap_d, tmap_x, ids, slots, pv, zws, group_counters, T, h_in, R_pad, n_slots, max_tokens, target_items,        \
            fill_warps, late_ticket, status)
  if (depth == 2) return a_q8 ? EDGELORA_SHRINK(2, true) : EDGELORA_SHRINK(2, false);
  return a_q8 ? EDGELORA_SHRINK(4, true) : EDGELORA_SHRINK(4, false);
#undef EDGELORA_SHRINK
}

}  // namespace edgelora
