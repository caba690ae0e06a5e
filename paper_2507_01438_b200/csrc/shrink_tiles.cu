// Shrink of a large batch on the tensor cores: z[t] = s_a A_a x[t] (paper Section 2.1 for A: r x h_in; Section
// 4.3: tokens that share an adapter are handled as one sub-batch), for one linear site or for a run of
// sites that see the same batch.
//
// D[128 x N] (fp32, in tensor memory) = R[128 x K] * C[N x K]^T from K blocks of 64, with two kinds of tiles:
//   segment tile  R = 128 tokens of a long run, C = A_a (N = R_pad): the run's tokens are contiguous in x;
//   gather tile   R = the A blocks of 128 / R_pad consecutive adapter groups stacked (one TMA box per group),
//                 C = the x rows of those groups' tokens, fetched four rows per gather copy; cross terms
//                 (adapter i times tokens of adapter j) are computed and never read.
// K is cut into `splits` parts per tile, each part writes its own plane of z, and whichever part arrives last
// adds the planes in order and writes the result; nobody waits for another CTA.  For the pair kernel the
// result is z in bf16, the operand of the expand: its builder threads read 16-byte chunks once, where adding
// up to eight fp32 planes per output tile kept them busy for 15 us of a 15 us tile (3080 -> 5000, rank 64).
// The items (tile, K part) of all sites form one list dealt round-robin to a persistent grid: what bounds an
// item is its chain of K blocks, so a launch that carries many sites is paid at the rate of its items instead
// of one ramp-up and one partial wave per site.
//
// Warp roles: warp 0 issues TMA, warp 1 owns tensor memory and issues the MMAs, warps 2..5 write z, warps
// 6..9 take their part of the copies of gather tiles.  Every mbarrier wait is bounded.
#include <algorithm>

#include "launch.cuh"
#include "ptx.cuh"
#include "shrink_tiles.h"
#include "tile_order.h"

namespace edgelora {

// Eight consecutive values of z, from rank index r0 on, as one 16-byte chunk of the operand: values at or past the
// true rank forced to zero.
__device__ __forceinline__ uint4 pack_z_chunk(const float (&v)[8], int32_t r0, int32_t rank) {
  float m[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) m[i] = r0 + i < rank ? v[i] : 0.f;
  return make_uint4(ptx::pack_bf16x2(m[0], m[1]), ptx::pack_bf16x2(m[2], m[3]), ptx::pack_bf16x2(m[4], m[5]),
                    ptx::pack_bf16x2(m[6], m[7]));
}

namespace {

static_assert(kTileGatherN == kGatherPass, "tokens of a pass");
constexpr int kThreads = 320;
constexpr uint32_t kRBytes = kTileM * kBlockK * 2;
constexpr uint32_t kStageBytes = kRBytes + kTileGatherN * kBlockK * 2;  // C: up to 64 rows (A_a, or gathered tokens)
constexpr int kAccCols = 64;

struct Barriers {
  uint64_t full[kTileStages];   // TMA -> MMA
  uint64_t empty[kTileStages];  // MMA -> TMA
  uint64_t zfull[kTileStages];  // the copy helpers have been through the stage -> MMA (gather tiles)
  uint64_t zgo[kTileStages];    // TMA warp -> copy helpers: the stage is free
  uint64_t tfull[2];            // MMA -> epilogue
  uint64_t tempty[2];           // epilogue -> MMA
  uint64_t ep;                  // rendezvous of the epilogue warps
  uint32_t tmem_slot;
  volatile uint32_t abort_flag;
  volatile int32_t last;        // this CTA's part of the tile arrived last
};
static_assert(sizeof(Barriers) <= kTileTailBytes, "tail of the shared memory");

struct Item {
  int32_t row, nrows, slot;    // segment tile: first token, tokens of the run in it, adapter slot
  int32_t gather;              // 0 segment, 1 gather
  int32_t g0, ng, tok0, ntok;  // gather tile: groups, and their tokens perm_short[tok0 .. tok0 + ntok)
  int32_t tile, split, splits, kb0, kb1;  // tile: index of its arrival counter
};

// The two choices below are made once per site and role, most of the time not at all, and kept out of line: four roles
// walk the items, and the fetch of their code is part of a launch of ten microseconds.
//
// K splits of the gather tiles when the host leaves the choice to the device (it does not know how
// many adapters a batch touches): the count up to 8 whose items fill whole waves of the grid best,
// each split keeping at least four K blocks.
__device__ __noinline__ int32_t choose_splits(int32_t kb_total, int32_t n_gt, int32_t grid) {
  int32_t best = 1;
  float best_eff = 0.f;
  for (int32_t sp = 1; sp <= 8 && kb_total / sp >= 4; ++sp) {
    if ((sp - 1) * ((kb_total + sp - 1) / sp) >= kb_total) continue;  // every split needs a K block
    const int32_t items = n_gt * sp, waves = (items + grid - 1) / grid;
    const float eff = waves > 0 ? static_cast<float>(items) / static_cast<float>(waves * grid) : 0.f;
    if (eff > best_eff + 0.02f) {
      best_eff = eff;
      best = sp;
    }
  }
  return best;
}
__device__ __noinline__ int32_t choose_parts(int32_t n_tok, int32_t n_gt, int32_t items, int32_t grid) {
  return gather_parts_lg(n_tok, n_gt, items, grid);
}

// Walks the items of all sites in order.
template <typename Batch>
struct Cursor {
  const Batch &b;
  int32_t s = -1, base = 0, n_items = 0;
  int32_t n_seg = 0, seg_splits = 1, n_gt = 0, g_splits = 1, lg_parts = 0;
  __device__ explicit Cursor(const Batch &batch) : b(batch) {}
  __device__ bool seek(int32_t item) {
    while (item >= base + n_items) {
      base += n_items;
      if (++s >= b.n_sites) return false;
      const ShrinkSite &st = b.site[s];
      const int32_t per = kTileM / st.R_pad;
      n_gt = (b.counts[4] + per - 1) / per;
      n_seg = st.splits > 0 ? b.counts[2] : 0;
      seg_splits = max(st.splits, 1);
      g_splits = st.splits > 0 ? st.splits : choose_splits(st.kb_total, n_gt, gridDim.x);
      const int32_t n_tok = st.splits > 0 ? b.counts[6] : 0;
      lg_parts = n_tok > kTileGatherN ? choose_parts(n_tok, n_gt, n_gt * g_splits * b.n_sites, gridDim.x) : 0;
      n_items = n_seg * seg_splits + (n_gt << lg_parts) * g_splits;
    }
    return true;
  }
  __device__ Item at(int32_t item) const {
    const ShrinkSite &st = b.site[s];
    Item c;
    int32_t local = item - base;
    c.row = c.nrows = c.slot = c.g0 = c.ng = c.tok0 = c.ntok = 0;
    if (local < n_seg * seg_splits) {
      c.gather = 0;
      c.tile = local % n_seg;
      c.split = local / n_seg;
      c.splits = seg_splits;
      c.row = b.sgmv_tiles[4 * c.tile + 0];
      c.nrows = b.sgmv_tiles[4 * c.tile + 1];
      c.slot = b.sgmv_tiles[4 * c.tile + 2];
      if (!EL_CHECK(st.status, c.row >= 0 && c.nrows >= 0 && c.row + c.nrows <= b.T && c.slot >= 0 && c.slot < b.n_slots, 4)) {
        c.row = 0;  // a tile of no rows: computed, nothing written
        c.nrows = 0;
        c.slot = 0;
      }
    } else {
      local -= n_seg * seg_splits;
      const int32_t n_tiles = n_gt << lg_parts;
      c.gather = 1;
      c.split = local / n_tiles;
      c.splits = g_splits;
      const int32_t t = local - c.split * n_tiles, g = t >> lg_parts;
      c.tile = n_seg + t;
      const int32_t per = kTileM / st.R_pad, n_groups = b.counts[0], n_lg = b.counts[4];
      c.g0 = (n_groups - n_lg) + g * per;  // the group of id -1, when there is one, comes first
      c.ng = min(per, n_groups - c.g0);
      c.tok0 = b.gs_short[c.g0];
      c.ntok = b.gs_short[c.g0 + c.ng] - c.tok0;
      if (lg_parts > 0) {
        const GatherPart part = gather_part(c.ntok, t - (g << lg_parts), lg_parts);
        c.tok0 += part.skip;
        c.ntok = part.n;
      }
    }
    const int32_t per_split = (st.kb_total + c.splits - 1) / c.splits;
    c.kb0 = min(c.split * per_split, st.kb_total);
    c.kb1 = min(st.kb_total, c.kb0 + per_split);
    return c;
  }
};
// Passes over a tile: a gather tile with more tokens than one pass holds takes several (none without tokens).
__device__ __forceinline__ int32_t passes_of(const Item &c) {
  return c.gather ? (c.ntok + kTileGatherN - 1) / kTileGatherN : 1;
}

// The copies of one pass over a gather tile, K blocks [kb0, kb1).  A K block needs one copy per
// group of the tile (its A block, R_pad rows of the R operand) and one per token quad (four rows of
// x into the C operand).  The copies of a K block are dealt out to kGatherParts warps (the producer warp is
// part 0 and also posts the byte count; the four helper warps are parts 1..4): copy i goes to part
// i % kGatherParts, looked up by lane i / kGatherParts.
// The parts other than the producer follow it: the producer announces a free stage on the stage's
// "go" barrier, every other part waits for that, issues its copies and arrives on the stage's
// "z full" barrier, which the MMA warp waits for beside the byte count.  (Waiting on the stage's
// empty barrier directly would not do: a part that has nothing to copy for a while can get several
// ring revolutions ahead, and a parity wait cannot tell revolutions apart.)  A copy that lands before
// the byte count is posted only drives the barrier's transaction count below zero for a moment.
constexpr int kGatherParts = 5;
constexpr int kGatherItems = (kTileM / 16 + kTileGatherN / 4 + kGatherParts - 1) / kGatherParts;  // copies of a part
template <typename Batch>
__device__ __forceinline__ bool gather_pass_copies(const Batch &b, const ShrinkSite &st, const Item &tc, int32_t t0,
                                                   uint8_t *smem, Barriers &sh, int part, int lane, uint32_t &stage,
                                                   uint32_t &phase, uint32_t &gophase) {
  const CUtensorMap *mg = &b.xg[st.x_index];
  const uint32_t a_bytes = static_cast<uint32_t>(st.R_pad) * kBlockK * 2;
  const int32_t n = min(kTileGatherN, tc.ntok - t0);
  const int32_t n_quads = (n + 3) >> 2;
  // live groups of the tile (an empty slot has no A block to fetch), for the byte count
  int32_t slot_l = -1;
  if (lane < tc.ng) {
    const int32_t a = b.group_adapter[tc.g0 + lane];
    if (a >= 0 && st.slots[a].rank > 0) slot_l = a;
  }
  const uint32_t live_mask = __ballot_sync(0xffffffffu, slot_l >= 0);
  const uint32_t tx = __popc(live_mask) * a_bytes + static_cast<uint32_t>(n_quads) * 4 * kBlockK * 2;
  // this lane's copy
  const int32_t item = part + kGatherParts * lane;
  int32_t my_slot = -1, my_quad = -1, tok[4] = {0, 0, 0, 0};
  const int32_t slot_of_item = __shfl_sync(0xffffffffu, slot_l, item < tc.ng ? item : 0);
  if (item < tc.ng) {
    my_slot = slot_of_item;
  } else if (item - tc.ng < n_quads) {
    my_quad = item - tc.ng;
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // rows past the pass's last token repeat it (they land in unused columns)
      tok[i] = b.perm_short[tc.tok0 + t0 + min(my_quad * 4 + i, n - 1)];
      if (!EL_CHECK(st.status, tok[i] >= 0 && tok[i] < b.T, 5)) tok[i] = 0;
    }
  }
  // One thread walks the K blocks and issues all of the part's copies (lane after lane, a warp-wide issue cost a
  // hundred cycles per copy): it takes over what the lanes have looked up.
  int32_t slot_j[kGatherItems], quad_j[kGatherItems], tok_j[kGatherItems][4];
#pragma unroll
  for (int j = 0; j < kGatherItems; ++j) {
    slot_j[j] = __shfl_sync(0xffffffffu, my_slot, j);
    quad_j[j] = __shfl_sync(0xffffffffu, my_quad, j);
#pragma unroll
    for (int i = 0; i < 4; ++i) tok_j[j][i] = __shfl_sync(0xffffffffu, tok[i], j);
  }
  const bool issuer = ptx::elect_one() != 0;
  const int src = __ffs(__ballot_sync(0xffffffffu, issuer)) - 1;
  int good = 1;
  if (issuer) {
    for (int32_t kb = tc.kb0; kb < tc.kb1; ++kb) {
      const bool got = part == 0 ? ptx::mbar_wait(&sh.empty[stage], phase ^ 1, b.wait_cycles)
                                 : ptx::mbar_wait(&sh.zgo[stage], (gophase >> stage) & 1u, b.wait_cycles);
      if (!got || sh.abort_flag) {
        good = 0;
        break;
      }
      gophase ^= 1u << stage;
      uint8_t *sr = smem + static_cast<size_t>(stage) * kStageBytes;
      if (part == 0) {
        ptx::mbar_arrive(&sh.zgo[stage]);
        ptx::mbar_arrive_expect_tx(&sh.full[stage], tx);
      }
#pragma unroll
      for (int j = 0; j < kGatherItems; ++j) {
        if (slot_j[j] >= 0)
          ptx::tma_load_2d(sr + static_cast<size_t>(part + kGatherParts * j) * a_bytes, &st.a, &sh.full[stage],
                           kb * kBlockK, slot_j[j] * st.R_pad);
        if (quad_j[j] >= 0)
          ptx::tma_gather4_2d(sr + kRBytes + static_cast<size_t>(quad_j[j]) * (4 * kBlockK * 2), mg, &sh.full[stage],
                              kb * kBlockK, tok_j[j][0], tok_j[j][1], tok_j[j][2], tok_j[j][3]);
      }
      if (part != 0) ptx::mbar_arrive(&sh.zfull[stage]);
      if (++stage == kTileStages) {
        stage = 0;
        phase ^= 1;
      }
    }
  }
  stage = __shfl_sync(0xffffffffu, stage, src);
  phase = __shfl_sync(0xffffffffu, phase, src);
  gophase = __shfl_sync(0xffffffffu, gophase, src);
  return __shfl_sync(0xffffffffu, good, src) != 0;
}

}  // namespace

template <int kSites>
__global__ void __launch_bounds__(kThreads, 1) shrink_tiles_kernel(const __grid_constant__ ShrinkBatch<kSites> b) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  Barriers &sh = *reinterpret_cast<Barriers *>(smem + static_cast<size_t>(kTileStages) * kStageBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long wl = b.wait_cycles;

  if (threadIdx.x == 0) {
    ptx::prefetch_tensormap(&b.x[b.site[0].x_index]);
    ptx::prefetch_tensormap(&b.xg[b.site[0].x_index]);
    ptx::prefetch_tensormap(&b.site[0].a);
    for (int s = 0; s < kTileStages; ++s) {
      ptx::mbar_init(&sh.full[s], 1);
      ptx::mbar_init(&sh.empty[s], 1);
      ptx::mbar_init(&sh.zfull[s], 4);  // one arrival per helper warp
      ptx::mbar_init(&sh.zgo[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&sh.tfull[i], 1);
      ptx::mbar_init(&sh.tempty[i], 4);  // one arrival per epilogue warp
    }
    ptx::mbar_init(&sh.ep, 4);
    sh.abort_flag = 0;
    ptx::fence_barrier_init();
  }
  if (warp == 1) {
    ptx::tmem_alloc(&sh.tmem_slot, 2 * kAccCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = sh.tmem_slot;
  ptx::pdl_launch_dependents();
  ptx::pdl_wait_prior_grids();  // the tile lists come from the plan kernel; earlier kernels may still read z

  Cursor<ShrinkBatch<kSites>> cur(b);
  const int32_t grid = static_cast<int32_t>(gridDim.x);
  bool ok = true;
  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    // The whole warp walks the loop: one thread issues the tile loads of a segment tile, and for gather
    // tiles every lane issues its share of the copies.
    uint32_t stage = 0, phase = 0, unused_go = 0;
    for (int32_t item = blockIdx.x; ok && cur.seek(item); item += grid) {
      const ShrinkSite &st = b.site[cur.s];
      const Item tc = cur.at(item);
      if (tc.gather) {
        for (int32_t t0 = 0; ok && t0 < tc.ntok; t0 += kTileGatherN)
          ok = gather_pass_copies(b, st, tc, t0, smem, sh, 0, lane, stage, phase, unused_go);
        continue;
      }
      const uint32_t tx_bytes = kRBytes + static_cast<uint32_t>(st.R_pad) * kBlockK * 2;
      const uint32_t stage0 = stage, phase0 = phase;
      bool good = true;
      if (ptx::elect_one()) {
        uint32_t sg = stage0, ph = phase0;
        for (int32_t kb = tc.kb0; kb < tc.kb1; ++kb) {
          if (!ptx::mbar_wait(&sh.empty[sg], ph ^ 1, wl) || sh.abort_flag) {
            good = false;
            break;
          }
          uint8_t *sr = smem + static_cast<size_t>(sg) * kStageBytes;
          ptx::mbar_arrive_expect_tx(&sh.full[sg], tx_bytes);
          ptx::tma_load_2d(sr, &b.x[st.x_index], &sh.full[sg], kb * kBlockK, tc.row);
          ptx::tma_load_2d(sr + kRBytes, &st.a, &sh.full[sg], kb * kBlockK, tc.slot * st.R_pad);
          if (++sg == kTileStages) {
            sg = 0;
            ph ^= 1;
          }
        }
      }
      ok = __all_sync(0xffffffffu, good);
      const uint32_t pos = stage0 + static_cast<uint32_t>(tc.kb1 - tc.kb0);
      stage = pos % kTileStages;
      phase = phase0 ^ ((pos / kTileStages) & 1u);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (ptx::elect_one()) {
      uint32_t stage = 0, phase = 0, zphase = 0;  // zphase: one parity bit per stage
      int32_t it = 0;
      for (int32_t item = blockIdx.x; ok && cur.seek(item); item += grid) {
        const ShrinkSite &st = b.site[cur.s];
        const Item tc = cur.at(item);
        const int32_t n_pass = passes_of(tc);
        for (int32_t pass = 0; ok && pass < n_pass; ++pass, ++it) {
          // UMMA N: the rank stride, or for a gather pass its token count rounded up to 16
          const uint32_t n_cols =
              tc.gather ? static_cast<uint32_t>((min(kTileGatherN, tc.ntok - pass * kTileGatherN) + 15) & ~15)
                        : static_cast<uint32_t>(st.R_pad);
          const uint32_t idesc = ptx::umma_idesc_bf16(kTileM, n_cols);
          const uint32_t acc = it & 1;
          if (!ptx::mbar_wait(&sh.tempty[acc], ((it >> 1) & 1) ^ 1, wl) || sh.abort_flag) {
            ok = false;
            break;
          }
          ptx::tc_fence_after_sync();
          const uint32_t tmem_d = tmem_base + acc * kAccCols;
          for (int32_t kb = tc.kb0; kb < tc.kb1; ++kb) {
            if (!ptx::mbar_wait(&sh.full[stage], phase, wl) || sh.abort_flag) {
              ok = false;
              break;
            }
            if (tc.gather) {  // the other parts of the tile's copies have been through this stage
              if (!ptx::mbar_wait(&sh.zfull[stage], (zphase >> stage) & 1u, wl)) {
                ok = false;
                break;
              }
              zphase ^= 1u << stage;
            }
            ptx::tc_fence_after_sync();
            const uint32_t sr = ptx::smem_u32(smem + static_cast<size_t>(stage) * kStageBytes);
            const uint64_t da = ptx::umma_desc_k128(sr), db = ptx::umma_desc_k128(sr + kRBytes);
#pragma unroll
            for (int k = 0; k < kBlockK / kUmmaK; ++k)
              ptx::umma_bf16(tmem_d, da + 2 * k, db + 2 * k, idesc, (kb > tc.kb0 || k > 0) ? 1u : 0u);
            ptx::umma_commit(&sh.empty[stage]);
            if (++stage == kTileStages) {
              stage = 0;
              phase ^= 1;
            }
          }
          if (ok) ptx::umma_commit(&sh.tfull[acc]);
        }
      }
    }
  } else if (warp < 6) {
    // ------------------------------------------------------------ epilogue: z (warps 2..5)
    const int quad = warp & 3, row_in_tile = quad * 32 + lane, etid = threadIdx.x - 64;
    int32_t it = 0;
    uint32_t ep_phase = 0;
    // the four warps meet on a barrier with a bounded wait, like every wait of this kernel
    auto ep_sync = [&]() {
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&sh.ep);
      const bool met = __all_sync(0xffffffffu, ptx::mbar_wait(&sh.ep, ep_phase, wl));
      ep_phase ^= 1u;
      return met;
    };
    for (int32_t item = blockIdx.x; ok && cur.seek(item); item += grid) {
      const ShrinkSite &st = b.site[cur.s];
      const Item tc = cur.at(item);
      const int32_t R = st.R_pad;
      const size_t plane = static_cast<size_t>(st.max_tokens) * R;
      float *zsplit = st.zws + static_cast<size_t>(tc.split) * plane;
      auto wait_acc = [&](uint32_t acc) {
        return __all_sync(0xffffffffu, ptx::mbar_wait(&sh.tfull[acc], (it >> 1) & 1, wl) && !sh.abort_flag);
      };
      if (tc.gather) {
        // accumulator row m = (group m / R of the tile, rank row m % R), column c = token
        // perm_short[tok0 + pass * 64 + c].  This thread writes z of its rank row for the tokens of its
        // group, scaled by s_a.
        const int32_t gi = row_in_tile / R, r = row_in_tile % R;
        int32_t c_lo = 0, c_hi = 0;  // this row's tokens, as positions inside the tile's token list
        float scale = 0.f;
        bool live = false;
        if (gi < tc.ng) {
          const SlotRow row = st.slots[b.group_adapter[tc.g0 + gi]];
          live = row.rank > 0;
          scale = row.scale;
          c_lo = b.gs_short[tc.g0 + gi] - tc.tok0;
          c_hi = b.gs_short[tc.g0 + gi + 1] - tc.tok0;
        }
        const int32_t n_pass = passes_of(tc);
        for (int32_t pass = 0; ok && pass < n_pass; ++pass, ++it) {
          const uint32_t acc = it & 1;
          ok = wait_acc(acc);
          if (!ok) break;
          ptx::tc_fence_after_sync();
          const int32_t t0 = pass * kTileGatherN, n = min(kTileGatherN, tc.ntok - t0);
          int32_t tok[2];  // lane l keeps the tokens of columns l and l + 32
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int c = q * 32 + lane;
            tok[q] = c < n ? b.perm_short[tc.tok0 + t0 + c] : 0;
            if (!EL_CHECK(st.status, tok[q] >= 0 && tok[q] < st.max_tokens, 6)) tok[q] = 0;
          }
          const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + acc * kAccCols;
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int32_t c0 = q * 32;
            if (c0 < n) {  // uniform over the warp (the columns past the tokens are never stored)
              float v[32];
              ptx::tmem_ld_32x32(taddr + c0, v);
#pragma unroll
              for (int jj = 0; jj < 32; ++jj) {
                const int32_t t = __shfl_sync(0xffffffffu, tok[q], jj);
                const int32_t c = t0 + c0 + jj;  // position inside the tile's token list
                if (live && c >= c_lo && c < c_hi && c0 + jj < n) zsplit[static_cast<size_t>(t) * R + r] = scale * v[jj];
              }
            }
          }
          ptx::tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&sh.tempty[acc]);
        }
        if (!ok) break;
      } else {
        // segment tile: row = token of the run, columns = rank index; z partial = scale * acc
        const uint32_t acc = it & 1;
        const float scale = st.slots[tc.slot].scale;
        ok = wait_acc(acc);
        if (!ok) break;
        ++it;
        ptx::tc_fence_after_sync();
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + acc * kAccCols;
        float *zrow = zsplit + static_cast<size_t>(tc.row + row_in_tile) * R;
        for (int c0 = 0; c0 < R; c0 += 32) {
          float v[32];
          ptx::tmem_ld_32x32(taddr + c0, v);  // (with a rank stride of 16 the second half is not stored)
          if (row_in_tile < tc.nrows)
#pragma unroll
            for (int q = 0; q < 32; q += 4)
              if (c0 + q < R)
                *reinterpret_cast<float4 *>(zrow + c0 + q) =
                    make_float4(scale * v[q], scale * v[q + 1], scale * v[q + 2], scale * v[q + 3]);
        }
        ptx::tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&sh.tempty[acc]);
      }
      // The part that arrives last adds the planes of all parts, in order, eight values per thread.
      __threadfence();  // this thread's z stores, before the arrival below
      if (!(ok = ep_sync())) break;
      if (etid == 0) {
        const int32_t old = tc.splits > 1 ? atomicAdd(&st.tile_counters[tc.tile], 1) : 0;
        sh.last = (old == tc.splits - 1) ? 1 : 0;
        if (tc.splits > 1 && old == tc.splits - 1) st.tile_counters[tc.tile] = 0;  // ready for the next launch
      }
      if (!(ok = ep_sync())) break;
      if (sh.last) {
        __threadfence();
        // Four chunks of eight values per thread and round, their loads of a plane in flight together: with one
        // chunk at a time the sum of seven planes of 128 x 64 took 20 us.
        const int nch = R >> 3, n_chunks = (tc.gather ? tc.ntok : tc.nrows) * nch;
        float *out = st.zws + static_cast<size_t>(kMaxZSplits) * plane;
        for (int i0 = etid; i0 < n_chunks; i0 += 4 * 128) {
          int32_t tok[4], rank[4];
          float acc[4][8];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int i = i0 + q * 128, k = i / nch;
            tok[q] = i < n_chunks ? (tc.gather ? b.perm_short[tc.tok0 + k] : tc.row + k) : -1;
            if (!EL_CHECK(st.status, tok[q] < b.T, 7)) tok[q] = -1;
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            rank[q] = 0;  // nothing loaded: nobody reads this z
            if (tok[q] >= 0) rank[q] = st.slots[tc.gather ? b.ids_valid[tok[q]] : tc.slot].rank;
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[q][e] = 0.f;
          }
#pragma unroll 2
          for (int32_t sp = 0; sp < tc.splits; ++sp) {
            float4 u[4], w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int c = (i0 + q * 128) % nch;
              const float4 *zp = reinterpret_cast<const float4 *>(st.zws + sp * plane + static_cast<size_t>(max(tok[q], 0)) * R + c * 8);
              u[q] = tok[q] >= 0 ? __ldcg(zp) : make_float4(0.f, 0.f, 0.f, 0.f);
              w[q] = tok[q] >= 0 ? __ldcg(zp + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              acc[q][0] += u[q].x; acc[q][1] += u[q].y; acc[q][2] += u[q].z; acc[q][3] += u[q].w;
              acc[q][4] += w[q].x; acc[q][5] += w[q].y; acc[q][6] += w[q].z; acc[q][7] += w[q].w;
            }
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (rank[q] <= 0) {
              if (tok[q] >= 0) atomicOr(st.status, EDGELORA_STATUS_SLOT_EMPTY);
              continue;
            }
            const int c = (i0 + q * 128) % nch;
            if (b.z_bf16) {
              reinterpret_cast<uint4 *>(out)[static_cast<size_t>(tok[q]) * nch + c] = pack_z_chunk(acc[q], c * 8, rank[q]);
            } else {
              float4 *o = reinterpret_cast<float4 *>(out + static_cast<size_t>(tok[q]) * R + c * 8);
              o[0] = make_float4(acc[q][0], acc[q][1], acc[q][2], acc[q][3]);
              o[1] = make_float4(acc[q][4], acc[q][5], acc[q][6], acc[q][7]);
            }
          }
        }
      }
      if (!(ok = ep_sync())) break;  // `last` is reused by the next tile
    }
  } else {
    // ------------------------------------------------------------ copy helpers (warps 6..9)
    uint32_t count = 0, gophase = 0;  // K blocks so far: stage = count % stages; one parity bit per stage
    for (int32_t item = blockIdx.x; ok && cur.seek(item); item += grid) {
      const ShrinkSite &st = b.site[cur.s];
      const Item tc = cur.at(item);
      if (!tc.gather) {
        count += static_cast<uint32_t>(tc.kb1 - tc.kb0);
        continue;
      }
      for (int32_t t0 = 0; ok && t0 < tc.ntok; t0 += kTileGatherN) {
        uint32_t stage = count % kTileStages, phase = 0;
        ok = gather_pass_copies(b, st, tc, t0, smem, sh, warp - 5, lane, stage, phase, gophase);
        count += static_cast<uint32_t>(tc.kb1 - tc.kb0);
      }
    }
  }
  if (!ok) {  // the items that this CTA leaves undone may belong to any site, and leave its arrival counters short
    sh.abort_flag = 1;
    for (int32_t s = 0; s < b.n_sites; ++s) atomicOr(b.site[s].status, EDGELORA_STATUS_TIMEOUT);
    ptx::settle();
  }
  __syncwarp();
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tmem_base, 2 * kAccCols);
  }
}

constexpr size_t kShrinkTilesSmem = 1024 + static_cast<size_t>(kTileStages) * kStageBytes + kTileTailBytes;

cudaError_t shrink_tiles_set_smem_limit() {
  const int bytes = static_cast<int>(kShrinkTilesSmem);
  cudaError_t e = cudaFuncSetAttribute(shrink_tiles_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(shrink_tiles_kernel<kTileSites>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e;
}

template <int kSites>
cudaError_t launch_shrink_tiles(const ShrinkBatch<kSites> &b, int32_t grid, bool pdl, cudaStream_t stream) {
  return launch_ex(shrink_tiles_kernel<kSites>, dim3(grid), dim3(kThreads), kShrinkTilesSmem, stream, pdl, 1, b);
}
template cudaError_t launch_shrink_tiles<1>(const ShrinkBatch<1> &, int32_t, bool, cudaStream_t);
template cudaError_t launch_shrink_tiles<kTileSites>(const ShrinkBatch<kTileSites> &, int32_t, bool, cudaStream_t);

}  // namespace edgelora
