// Base product and expand of a large batch on CTA pairs (paper Section 3.4: the base product is batched
// over every token, the low-rank expand B_a z is folded into the same accumulator, y is written once),
// for one linear site or for a run of sites that see the same batch.
//
// y[256 tokens x BN] = x[256 x K] * W[BN x K]^T per tile, K blocks of 64, one tile per pair of CTAs (two
// SMs of a cluster): tcgen05.mma.cta_group::2 multiplies operands that lie half in one CTA's shared memory
// and half in the other's.  CTA c of the pair holds the tokens [128 c, 128 c + 128) of the tile and the W
// rows [c BN/2, (c + 1) BN/2), so a K block costs an SM 32 KB of operand fill for 512 tensor cycles where
// a tile of 128 x 256 per SM costs 48 KB (4096 -> 14336, T = 4096: 289 us, 1.66 PFLOP/s, against 371 us; the tensor
// pipe is busy 87 % of the cycles, and what bounds a loop of calls is the power limit).  After the K blocks of h_in come
// the LoRA K blocks for the adapters of the tile's 256 tokens, 64 / R_pad adapters in a block: B_a rows (TMA, each CTA
// its half) against z in bf16 (each CTA writes the rows of its own tokens), where the MMA of an adapter adds to the
// accumulator rows of its tokens only.
//
// Warp roles, in both CTAs: warp 0 issues TMA, warp 1 owns tensor memory (and, in CTA 0 only, issues the
// MMAs of the pair), warps 2..5 are the epilogue of the CTA's 128 tokens, warps 6..9 list the tile's adapters
// and build the z operand.  Barriers that the MMA thread waits for live in CTA 0: the loads of both CTAs are
// counted on its "full" barriers, the builder and epilogue warps of CTA 1 arrive there remotely; commits
// arrive in both CTAs.  Every mbarrier wait is bounded; on a timeout the status word gets
// EDGELORA_STATUS_TIMEOUT and all roles leave their loops.
//
// The tiles of all sites of a launch form one list, one cluster of the grid per tile, so only the last wave of
// the whole list is partly empty instead of the last wave of every site.  The clusters that are resident first
// stay: while a pair works on a tile it takes the next cluster that has not started off the launch queue
// (cluster launch control).  Dealt out statically, pairs drifted apart (tiles with many adapters are half as
// long again) until the pairs that share a W or x tile no longer met in L2: a set of 28 sites at T = 2112 read
// 7.6 GB of DRAM for 2.1 GB of operands and paid for it in clock rate under the power limit (2.9 GB now).
#include "internal.cuh"
#include "launch.cuh"
#include "prefill.h"
#include "ptx.cuh"
#include "tile_order.h"

namespace edgelora {

namespace {

constexpr int kThreads = 320;
constexpr uint32_t kXBytes = kTileM * kBlockK * 2;  // a CTA's half of the token operand: 16 KB
constexpr int kListMax = kListTile;                 // adapters of a tile at most

struct Barriers {
  uint64_t full[kPairMaxStages];   // CTA 0: loads of both CTAs -> MMA
  uint64_t empty[kPairMaxStages];  // MMA -> TMA (own CTA)
  uint64_t zfull[kPairMaxStages];  // CTA 0: builder warps of CTA 1 -> MMA: their rows of z (first LoRA K blocks of a tile)
  uint64_t mfull[kPairMaxStages];  // builder -> MMA (own CTA): whose rows the LoRA K block is for, and CTA 0's rows of z
  uint64_t zgo[kPairMaxStages];    // TMA warp -> builder (own CTA): the stage is free
  uint64_t tfull[2];               // MMA -> epilogue (own CTA)
  uint64_t tempty[2];              // CTA 0: epilogue warps of both CTAs -> MMA
  uint64_t lfull[2];               // builder -> TMA, MMA: the tile's adapter list is written
  uint64_t lempty[2];              // TMA, MMA -> builder
  uint64_t nfull;                  // the answer that names the next tile has arrived
  uint64_t nempty;                 // CTA 1: every role of both CTAs has read it
  uint64_t ask;                    // CTA 1: its TMA thread is near the end of the tile's K blocks
  alignas(16) uint32_t answer[4];
  // CTA 0: per adapter of a LoRA K block, the rows of the tile that are not on it
  alignas(16) uint32_t off[kPairMaxStages][kBlockK / kUmmaK][8];
  uint32_t tmem_slot;
  volatile uint32_t abort_flag;
  int32_t wcount[8];
  int32_t count[2];
  int32_t list[2][kListMax];
};
static_assert(sizeof(Barriers) <= kPairTailBytes, "tail of the shared memory");

__device__ __forceinline__ void named_bar(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// The same barrier; every thread learns whether any of them passed true.
__device__ __forceinline__ bool named_bar_any(int id, int threads, bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %3, 0;\n\tbar.red.or.pred q, %1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(id), "r"(threads), "r"(v ? 1u : 0u)
      : "memory");
  return r != 0;
}

// What every role does between two tiles: the answer of the launch queue is read and handed back to the thread
// that asks (`nempty`: its barrier's cluster address), by whole warps (kWarp: one arrival per warp) or by single
// threads.  `tile` becomes the next tile, -1 when none is left.  Returns false when the wait ran out.
// Without kSteal the tiles are dealt round-robin to the pairs of the grid.
template <bool kWarp, bool kSteal>
__device__ __forceinline__ bool next_tile(Barriers &sh, int32_t it, uint32_t nempty, int32_t n_tiles, long long wl,
                                          int32_t &tile) {
  if (!kSteal) {
    tile += static_cast<int32_t>(gridDim.x >> 1);
    if (tile >= n_tiles) tile = -1;
    return true;
  }
  const bool got = ptx::mbar_wait_cluster(&sh.nfull, it & 1, wl);
  const int32_t cta = got ? ptx::cluster_taken(sh.answer) : -1;
  tile = cta < 0 ? -1 : cta >> 1;
  ptx::fence_proxy_async();  // the next answer is written through the async proxy
  if (kWarp) __syncwarp();
  if (!kWarp || (threadIdx.x & 31) == 0) ptx::mbar_arrive_cluster(nempty);
  return got;
}
// Adapters of a LoRA K block: 64 / R_pad (16, 32 or 64), without the division.
__device__ __forceinline__ int32_t lora_per(int32_t R_pad) { return kBlockK >> (31 - __clz(R_pad)); }
constexpr int kAnswerReaders = 10 + 9;  // TMA, MMA, 4 epilogue and 4 builder warps of CTA 0; CTA 1 issues no MMAs

}  // namespace

template <int kSites, bool kSteal>
__global__ void __launch_bounds__(kThreads, 1) pair_gemm_kernel(const __grid_constant__ PairBatch<kSites> b) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t w_bytes = static_cast<uint32_t>(b.BN) * (kBlockK * 2) / 2;  // a CTA's half of the W operand
  const uint32_t stage_bytes = kXBytes + w_bytes;
  const uint32_t nstages = static_cast<uint32_t>(b.stages);
  uint8_t *y_stage = smem + static_cast<size_t>(nstages) * stage_bytes;  // 4 KB per epilogue warp
  Barriers &sh = *reinterpret_cast<Barriers *>(y_stage + kYStageBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_rank();
  const bool leader = rank == 0;
  const int32_t tile0 = static_cast<int32_t>(blockIdx.x >> 1), n_tiles = b.site[b.n_sites - 1].tile_end;
  const long long wl = b.wait_cycles;

  if (threadIdx.x == 0) {
    ptx::prefetch_tensormap(&b.x[b.site[0].x_index]);
    ptx::prefetch_tensormap(&b.site[0].w);
    for (uint32_t s = 0; s < nstages; ++s) {
      ptx::mbar_init(&sh.full[s], 1);
      ptx::mbar_init(&sh.empty[s], 1);
      ptx::mbar_init(&sh.zfull[s], 4);  // one arrival per builder warp of CTA 1
      ptx::mbar_init(&sh.mfull[s], 4);  // one arrival per builder warp
      ptx::mbar_init(&sh.zgo[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&sh.tfull[i], 1);
      ptx::mbar_init(&sh.tempty[i], 8);  // one arrival per epilogue warp of the pair
      ptx::mbar_init(&sh.lfull[i], 1);
      ptx::mbar_init(&sh.lempty[i], leader ? 2 : 1);
    }
    ptx::mbar_init(&sh.nfull, 1);
    ptx::mbar_init(&sh.nempty, kAnswerReaders);
    ptx::mbar_init(&sh.ask, 1);
    sh.abort_flag = 0;
    ptx::fence_barrier_init();
  }
  if (warp == 1) {
    ptx::tmem_alloc_pair(&sh.tmem_slot, 512);
    ptx::tmem_relinquish_pair();
  }
  __syncwarp();
  ptx::tc_fence_before_sync();
  ptx::cluster_sync_all();  // the other CTA's barriers exist from here on
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = sh.tmem_slot;
  ptx::pdl_launch_dependents();

  const uint32_t nempty1 = ptx::map_to_rank(ptx::smem_u32(&sh.nempty), 1);
  bool ok = true;
  int32_t site = 0;
  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    // The base K blocks read x and W, which no kernel of this call writes: they start before the kernels
    // in front of this one (plan, shrink) are done.
    if (ptx::elect_one()) {
      uint32_t stage = 0, phase = 0, used = 0;
      int32_t it = 0;
      const uint32_t full0 = ptx::map_to_rank(ptx::smem_u32(&sh.full[0]), 0);
      auto wait_empty = [&]() { return ptx::mbar_wait(&sh.empty[stage], phase ^ 1, wl) && !sh.abort_flag; };
      auto advance = [&]() {
        ++used;
        if (++stage == nstages) {
          stage = 0;
          phase ^= 1;
        }
      };
      for (int32_t tile = tile0; tile >= 0; ++it) {
        const Tile t = tile_at(b, tile, site);
        const PairSite &st = b.site[t.s];
        const CUtensorMap *mx = &b.x[st.x_index];
        const int32_t row_x = t.m * (2 * kTileM) + static_cast<int32_t>(rank) * kTileM;
        const int32_t row_w = t.n * b.BN + static_cast<int32_t>(rank) * (b.BN / 2);
        const int32_t kb_ask = max(0, st.kb_total - kPairMaxStages);
        for (int32_t kb = 0; kb < st.kb_total; ++kb) {
          if (!wait_empty()) {
            ok = false;
            break;
          }
          if (kSteal && !leader && kb == kb_ask) ptx::mbar_arrive(&sh.ask);
          uint8_t *sr = smem + static_cast<size_t>(stage) * stage_bytes;
          const uint32_t bar = full0 + stage * 8;
          if (leader) ptx::mbar_arrive_expect_tx(&sh.full[stage], 2 * (kXBytes + w_bytes));
          ptx::tma_load_2d_pair(sr, mx, bar, kb * kBlockK, row_x);
          ptx::tma_load_2d_pair(sr + kXBytes, &st.w, bar, kb * kBlockK, row_w);
          advance();
        }
        if (!ok) break;
        const int buf = it & 1;
        if (!ptx::mbar_wait(&sh.lfull[buf], (it >> 1) & 1, wl)) {
          ok = false;
          break;
        }
        const int32_t cnt = sh.count[buf];
        const int32_t per = lora_per(st.R_pad);  // adapters of a LoRA K block
        const uint32_t b_bytes = static_cast<uint32_t>(b.BN * st.R_pad);  // a CTA's half of one adapter's rows
        for (int32_t e0 = 0, blk = 0; e0 < cnt; e0 += per, ++blk) {
          const int32_t n = min(per, cnt - e0);
          if (!wait_empty()) {
            ok = false;
            break;
          }
          // The stage is free: let the builder write its half (it follows this warp, never the stage
          // barriers directly, so it cannot run ahead of the ring).
          if (leader || blk < static_cast<int32_t>(nstages)) ptx::mbar_arrive(&sh.zgo[stage]);
          if (leader) ptx::mbar_arrive_expect_tx(&sh.full[stage], 2 * n * b_bytes);
          uint8_t *dst = smem + static_cast<size_t>(stage) * stage_bytes + kXBytes;
          for (int32_t j = 0; j < n; ++j)
            ptx::tma_load_3d_pair(dst + j * b_bytes, &st.b, full0 + stage * 8, 0, row_w, sh.list[buf][e0 + j]);
          advance();
        }
        if (!ok) break;
        ptx::mbar_arrive(&sh.lempty[buf]);
        ok = next_tile<false, kSteal>(sh, it, nempty1, n_tiles, wl, tile);
        if (!ok) break;
      }
      // the commits that hand the last stages back arrive in this CTA's shared memory: wait for them
      const RingPos last = ring_drain(used, nstages);
      stage = last.stage;
      phase = last.phase;
      for (uint32_t i = min(used, nstages); ok && i > 0; --i) {
        ok = ptx::mbar_wait(&sh.empty[stage], phase ^ 1, wl);
        advance();
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (of the pair)
    if (leader && ptx::elect_one()) {
      const uint32_t idesc = ptx::umma_idesc_bf16(2 * kTileM, static_cast<uint32_t>(b.BN));
      uint32_t stage = 0, phase = 0, zphase = 0, mphase = 0;  // zphase, mphase: one parity bit per stage
      int32_t it = 0;
      for (int32_t tile = tile0; tile >= 0; ++it) {
        const Tile t = tile_at(b, tile, site);
        const PairSite &st = b.site[t.s];
        const uint32_t acc = it & 1;
        if (!ptx::mbar_wait_cluster(&sh.tempty[acc], ((it >> 1) & 1) ^ 1, wl) || sh.abort_flag) {
          ok = false;
          break;
        }
        ptx::tc_fence_after_sync();
        const uint32_t tmem_d = tmem_base + acc * 256;
        auto commit = [&]() {  // frees the stage in both CTAs once its MMAs are done
          ptx::umma_commit_pair(&sh.empty[stage]);
          if (++stage == nstages) {
            stage = 0;
            phase ^= 1;
          }
        };
        for (int32_t kb = 0; kb < st.kb_total; ++kb) {
          if (!ptx::mbar_wait(&sh.full[stage], phase, wl) || sh.abort_flag) {
            ok = false;
            break;
          }
          ptx::tc_fence_after_sync();
          const uint32_t sr = ptx::smem_u32(smem + static_cast<size_t>(stage) * stage_bytes);
          const uint64_t da = ptx::umma_desc_k128(sr), db = ptx::umma_desc_k128(sr + kXBytes);
          // advancing 16 bf16 along K inside the swizzled row = 32 bytes = 2 descriptor units
#pragma unroll
          for (int k = 0; k < kBlockK / kUmmaK; ++k)
            ptx::umma_bf16_pair(tmem_d, da + 2 * k, db + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
          commit();
        }
        if (!ok) break;
        const int buf = it & 1;
        if (!ptx::mbar_wait(&sh.lfull[buf], (it >> 1) & 1, wl)) {
          ok = false;
          break;
        }
        const int32_t cnt = sh.count[buf];
        const int32_t per = lora_per(st.R_pad);
        const uint32_t b_bytes = static_cast<uint32_t>(b.BN * st.R_pad), row_bytes = static_cast<uint32_t>(st.R_pad) * 2;
        const int ksteps = st.R_pad >> 4;  // K steps of 16
        for (int32_t e0 = 0, blk = 0; e0 < cnt; e0 += per, ++blk) {
          const bool has_z = blk < static_cast<int32_t>(nstages);  // (later blocks find z in the stage, see the builder)
          if (!ptx::mbar_wait(&sh.full[stage], phase, wl) || !ptx::mbar_wait(&sh.mfull[stage], (mphase >> stage) & 1u, wl) ||
              (has_z && !ptx::mbar_wait_cluster(&sh.zfull[stage], (zphase >> stage) & 1u, wl)) || sh.abort_flag) {
            ok = false;
            break;
          }
          mphase ^= 1u << stage;
          if (has_z) zphase ^= 1u << stage;
          ptx::tc_fence_after_sync();
          const uint32_t sr = ptx::smem_u32(smem + static_cast<size_t>(stage) * stage_bytes);
          const uint64_t da = ptx::umma_desc_k128(sr);
          uint64_t db = ptx::umma_desc_rows(sr + kXBytes, row_bytes);
          const int32_t n = min(per, cnt - e0);
          for (int32_t j = 0; j < n; ++j, db += b_bytes >> 4) {
            const uint4 off_lo = *reinterpret_cast<const uint4 *>(&sh.off[stage][j][0]);
            const uint4 off_hi = *reinterpret_cast<const uint4 *>(&sh.off[stage][j][4]);
#pragma unroll
            for (int k = 0; k < kBlockK / kUmmaK; ++k)
              if (k < ksteps) ptx::umma_bf16_pair_rows(tmem_d, da + 2 * k, db + 2 * k, idesc, off_lo, off_hi);
          }
          commit();
        }
        if (!ok) break;
        ptx::mbar_arrive(&sh.lempty[buf]);
        ptx::umma_commit_pair(&sh.tfull[acc]);  // accumulator complete
        ok = next_tile<false, kSteal>(sh, it, nempty1, n_tiles, wl, tile);
        if (!ok) break;
      }
    } else if (kSteal && !leader && ptx::elect_one()) {
      // The pair's requests to the launch queue, one tile ahead: asked once every role has read the answer before,
      // and not before the loads of the tile at hand are nearly through (at the start of a launch clusters still
      // wait for their SMs; taking those tiles at once would leave the SMs that come free a moment later without
      // work).
      const uint32_t nfull0 = ptx::map_to_rank(ptx::smem_u32(&sh.nfull), 0);
      for (int32_t it = 0;; ++it) {
        if (!ptx::mbar_wait(&sh.ask, it & 1, wl) ||
            (it > 0 && !ptx::mbar_wait_cluster(&sh.nempty, (it - 1) & 1, wl)) || sh.abort_flag) {
          ok = false;
          break;
        }
        ptx::mbar_arrive_expect_tx(&sh.nfull, 16);
        ptx::mbar_arrive_expect_tx_cluster(nfull0, 16);
        ptx::cluster_try_cancel(sh.answer, &sh.nfull);
        if (!ptx::mbar_wait_cluster(&sh.nfull, it & 1, wl)) {
          ok = false;
          break;
        }
        if (ptx::cluster_taken(sh.answer) < 0) break;  // (after a refusal nothing more is asked)
        ptx::fence_proxy_async();
      }
    }
  } else if (warp < 6) {
    // ------------------------------------------------------------ epilogue (warps 2..5)
    const int quad = warp & 3;  // TMEM lanes [32 quad, 32 quad + 32) = this CTA's tokens 32 quad ..
    uint8_t *stage_rows = y_stage + quad * (32 * 128);
    const uint32_t tempty0 = ptx::map_to_rank(ptx::smem_u32(&sh.tempty[0]), 0);
    ptx::pdl_wait_prior_grids();  // earlier kernels may still read y
    int32_t it = 0;
    for (int32_t tile = tile0; tile >= 0; ++it) {
      const Tile t = tile_at(b, tile, site);
      const PairSite &st = b.site[t.s];
      const uint32_t acc = it & 1;
      const int32_t row0 = t.m * (2 * kTileM) + static_cast<int32_t>(rank) * kTileM + quad * 32;
      const int32_t col0 = t.n * b.BN;
      if (!__all_sync(0xffffffffu, ptx::mbar_wait(&sh.tfull[acc], (it >> 1) & 1, wl) && !sh.abort_flag)) {
        ok = false;
        break;
      }
      ptx::tc_fence_after_sync();
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + acc * 256;
      // lane = token, columns = output features.  64 columns at a time go to the warp's shared-memory stage as
      // bf16 (rows of 128 bytes, 16-byte chunks swizzled by the row so that the lanes' stores spread over the
      // banks) and leave as whole 128-byte lines, eight lanes per token.
      for (int32_t c0 = 0; c0 < b.BN; c0 += 64) {
        float v[64];
        ptx::tmem_ld_32x64(taddr + c0, v);  // (the tile may end 32 columns earlier: those values are not stored)
        if (c0 + 64 >= b.BN) {              // the accumulator is read: the next tile may have it
          ptx::tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive_cluster(tempty0 + acc * 8);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          uint4 o;
          o.x = ptx::pack_bf16x2(v[8 * q + 0], v[8 * q + 1]);
          o.y = ptx::pack_bf16x2(v[8 * q + 2], v[8 * q + 3]);
          o.z = ptx::pack_bf16x2(v[8 * q + 4], v[8 * q + 5]);
          o.w = ptx::pack_bf16x2(v[8 * q + 6], v[8 * q + 7]);
          *reinterpret_cast<uint4 *>(stage_rows + lane * 128 + ((q ^ (lane & 7)) << 4)) = o;
        }
        __syncwarp();
        const int ch = lane & 7;
        const int32_t col = col0 + c0 + ch * 8;  // h_out is a multiple of 8: a chunk is all in or all out
        const bool col_in = c0 + ch * 8 < b.BN && col < st.h_out;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = i * 4 + (lane >> 3);
          if (col_in && row0 + r < b.T)
            *reinterpret_cast<uint4 *>(st.y + static_cast<size_t>(row0 + r) * st.h_out + col) =
                *reinterpret_cast<const uint4 *>(stage_rows + r * 128 + ((ch ^ (r & 7)) << 4));
        }
        __syncwarp();
      }
      ok = __all_sync(0xffffffffu, next_tile<true, kSteal>(sh, it, nempty1, n_tiles, wl, tile));
      if (!ok) break;
    }
  } else {
    // ------------------------------------------------------------ adapter list and z operand (warps 6..9)
    const int btid = threadIdx.x - 192, bwarp = warp - 6;  // 0..127: one of the CTA's tokens
    const uint32_t zfull0 = ptx::map_to_rank(ptx::smem_u32(&sh.zfull[0]), 0);
    uint32_t count = 0;    // K blocks so far: stage = count % stages
    uint32_t gophase = 0;  // one parity bit per stage for zgo
    ptx::pdl_wait_prior_grids();  // tile lists and z come from the kernels before this one
    int32_t it = 0;
    for (int32_t tile = tile0; tile >= 0; ++it) {
      const Tile t = tile_at(b, tile, site);
      const PairSite &st = b.site[t.s];
      const int buf = it & 1;
      // The adapters of the tile whose slot is loaded, in the plan's order: worked out once per tile while
      // the base K blocks stream, so that the issuing threads find a list without gaps in shared memory
      // (following list entry -> slot row through global memory would cost them a microsecond per K block).
      // (All 128 threads come here for every tile and leave together, also when a wait of one of them ran out.)
      ok = ptx::mbar_wait(&sh.lempty[buf], ((it >> 1) & 1) ^ 1, wl) && !sh.abort_flag;
      if (named_bar_any(2, 128, !ok)) {
        ok = false;
        break;
      }
      const int32_t n_list = min(b.mt_count[t.m], kListMax);
      const int32_t tok = t.m * (2 * kTileM) + static_cast<int32_t>(rank) * kTileM + btid;
      int32_t id = tok < b.T ? b.ids_valid[tok] : -1;
      if (!EL_CHECK(st.status, id >= -1 && id < b.n_slots, 2)) id = -1;
      int32_t id1 = leader && tok + kTileM < b.T ? b.ids_valid[tok + kTileM] : -1;  // of a token of CTA 1
      if (!EL_CHECK(st.status, id1 >= -1 && id1 < b.n_slots, 2)) id1 = -1;
      // z of the thread's token, in flight while the list is made
      const int nch = st.R_pad >> 3;  // 16-byte chunks of one operand row that the MMAs read
      uint4 z[8];
#pragma unroll
      for (int c = 0; c < 8; ++c)
        z[c] = (id >= 0 && c < nch) ? __ldcg(st.zb + static_cast<size_t>(tok) * nch + c) : make_uint4(0u, 0u, 0u, 0u);
      int32_t mine[2];
      uint32_t live[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int e = h * 128 + btid;
        int32_t a = -1;
        if (e < n_list) {
          a = b.mt_list[t.m * kListMax + e];
          if (!EL_CHECK(st.status, a >= 0 && a < b.n_slots, 1)) a = -1;
          if (a >= 0 && st.slots[a].rank <= 0) a = -1;
        }
        mine[h] = a;
        live[h] = __ballot_sync(0xffffffffu, a >= 0);
        if (lane == 0) sh.wcount[h * 4 + bwarp] = __popc(live[h]);
      }
      named_bar(2, 128);
      int32_t before[2] = {0, 0}, total = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (i == bwarp) before[0] = total;
        if (i == 4 + bwarp) before[1] = total;
        total += sh.wcount[i];
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (mine[h] >= 0) sh.list[buf][before[h] + __popc(live[h] & ((1u << lane) - 1u))] = mine[h];
      if (btid == 0) sh.count[buf] = total;
      named_bar(2, 128);
      if (btid == 0) ptx::mbar_arrive(&sh.lfull[buf]);

      count += static_cast<uint32_t>(st.kb_total);
      // The MMA of an adapter multiplies the z of all tokens with its B, and the tensor core leaves the rows of the tokens
      // that are not on it as they are.  So z is the same for every block of the tile: it is written once per stage of
      // the ring, and what a block needs beyond that is eight words of rows per adapter.  It also keeps an infinity or NaN
      // in one adapter's B away from the tokens on others, which a product with zeros of z would not.  What bounds a tile
      // of many adapters is the hand-over of a stage with the latency of its B_a rows, hence 64 / R_pad adapters to a
      // stage: 300 tokens on 300 adapters of rank 16, 4096 -> 4096: 61 us, 115 with one adapter to a stage, 123 with z
      // masked and written anew for every adapter.
      const int32_t per = lora_per(st.R_pad);
      for (int32_t e0 = 0, blk = 0; e0 < total; e0 += per, ++blk) {
        const bool write_z = blk < static_cast<int32_t>(nstages);
        const uint32_t stage = count % nstages;
        ++count;
        if (!leader && !write_z) continue;
        ok = __all_sync(0xffffffffu, ptx::mbar_wait(&sh.zgo[stage], (gophase >> stage) & 1u, wl) && !sh.abort_flag);
        if (!ok) break;
        gophase ^= 1u << stage;
        if (write_z) {
          // 128-byte swizzle: the 16-byte chunk index is XORed with the row index modulo 8
          uint8_t *drow = smem + static_cast<size_t>(stage) * stage_bytes + btid * 128;
#pragma unroll
          for (int c = 0; c < 8; ++c)
            if (c < nch) *reinterpret_cast<uint4 *>(drow + ((c ^ (btid & 7)) << 4)) = z[c];
          ptx::fence_proxy_async();  // make the generic-proxy writes visible to the tensor core
        }
        if (leader) {
          for (int32_t j = 0; j < min(per, total - e0); ++j) {
            const int32_t a = sh.list[buf][e0 + j];
            const uint32_t on0 = __ballot_sync(0xffffffffu, id == a), on1 = __ballot_sync(0xffffffffu, id1 == a);
            if (lane == 0) {
              sh.off[stage][j][bwarp] = ~on0;
              sh.off[stage][j][4 + bwarp] = ~on1;
            }
          }
        }
        __syncwarp();
        if (lane == 0) {
          if (leader)
            ptx::mbar_arrive(&sh.mfull[stage]);
          else
            ptx::mbar_arrive_cluster(zfull0 + stage * 8);
        }
      }
      const bool got = next_tile<true, kSteal>(sh, it, nempty1, n_tiles, wl, tile);
      if (named_bar_any(2, 128, !ok || !got)) {
        ok = false;
        break;
      }
    }
  }
  if (!ok) {  // the tiles that this pair leaves undone may belong to any site
    sh.abort_flag = 1;
    for (int32_t s = 0; s < b.n_sites; ++s) atomicOr(b.site[s].status, EDGELORA_STATUS_TIMEOUT);
    ptx::settle();
  }
  __syncwarp();
  ptx::tc_fence_before_sync();
  ptx::cluster_sync_all();  // nothing of the other CTA touches this one's memory from here on
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc_pair(tmem_base, 512);
  }
}

static size_t pair_smem_bytes(int stages, int BN) {
  return 1024 + static_cast<size_t>(stages) * (kXBytes + BN * kBlockK) + kYStageBytes + kPairTailBytes;
}
int pair_stages(int BN) {
  const size_t fixed = 1024 + kYStageBytes + kPairTailBytes, stage = kXBytes + static_cast<size_t>(BN) * kBlockK;
  return std::min(kPairMaxStages, static_cast<int>((kPairSmemBudget - fixed) / stage));
}

cudaError_t pair_set_smem_limit() {
  const int bytes = static_cast<int>(kPairSmemBudget);
  cudaError_t e = cudaSuccess;
#define EDGELORA_SMEM(N, ST)                                                                                      \
  if (e == cudaSuccess) e = cudaFuncSetAttribute(pair_gemm_kernel<N, ST>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  EDGELORA_SMEM(1, false)
  EDGELORA_SMEM(1, true)
  EDGELORA_SMEM(kPairSites, false)
  EDGELORA_SMEM(kPairSites, true)
#undef EDGELORA_SMEM
  return e;
}

// Tiles come off the launch queue when the pairs run through more than four waves of them.  Shorter launches have no time
// to drift, and a kernel that uses the launch queue does not start under the tail of the kernel in front of it: 1 to 3 us
// per call in favour of the static deal up to four waves (4096 -> 6144, T = 2112, 2.9 waves: 96 against 99 us).  At five
// to seven waves the two differ by less than runs of one do (4096 -> 20480, T = 1024: 133-152 against 144-152 us), from
// nine on the queue is ahead (14 sites, T = 300: 398-459 against 428-536 us; T = 1024: 757-792 against 823-868 us).
template <int kSites>
cudaError_t launch_pair_gemm(const PairBatch<kSites> &b, int32_t sms, bool pdl, cudaStream_t stream) {
  const int32_t tiles = b.site[b.n_sites - 1].tile_end, grid = pair_grid(tiles, sms);
  const size_t smem = pair_smem_bytes(b.stages, b.BN);
  if (pair_queued(tiles, sms))
    return launch_ex(pair_gemm_kernel<kSites, true>, dim3(grid), dim3(kThreads), smem, stream, pdl, 2, b);
  return launch_ex(pair_gemm_kernel<kSites, false>, dim3(grid), dim3(kThreads), smem, stream, pdl, 2, b);
}
template cudaError_t launch_pair_gemm<1>(const PairBatch<1> &, int32_t, bool, cudaStream_t);
template cudaError_t launch_pair_gemm<kPairSites>(const PairBatch<kPairSites> &, int32_t, bool, cudaStream_t);

}  // namespace edgelora
