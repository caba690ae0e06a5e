// Small decode batches (at most 64 tokens) of batch LoRA inference (paper Section 3.4): the base product W [x_0 .. x_n] batched
// over every token, with the low-rank expand B_a z added in fp32 before y is written once; in the one-launch form the shrink
// too.  (Larger batches, or too few row tiles to split K: decode_tile.cu.  Runs of sites: decode_sites.cu.  Above 256 tokens:
// prefill.cu.)
//
// D[128 x BN] (fp32, in tensor memory) = R[128 x K] * C[BN x K]^T, both operands K-major bf16 in
// 128-byte-swizzled shared-memory tiles of 64 K elements ("K blocks"), multiplied by tcgen05.mma
// issued from one thread.  R = 128 rows of W, C = all tokens (N = T rounded up to 32 or 64).  W is streamed once; K is split
// across CTAs so every SM pulls from HBM.  The K splits of one row tile form a
// thread-block cluster: after the main loop every CTA sends its fp32 partial tile, column block by column
// block, into the shared memory of the CTA that owns those tokens (distributed shared memory), and each
// owner adds the partials in a fixed order, adds the expand of its tokens and writes its part of y.
//
// Warp roles: warp 0 issues TMA, warp 1 owns TMEM and issues the MMAs, warps 2..5 are the
// epilogue (each reads the 32 TMEM lanes of its quadrant), warps 6..9 the shrink team of a one-launch call.
// Every mbarrier wait is bounded; on a timeout the status word gets EDGELORA_STATUS_TIMEOUT and
// all roles leave their loops.
#include <cstdio>
#include <cstdlib>

#include "decode_route.cuh"
#include "expand.cuh"
#include "internal.cuh"
#include "launch.cuh"
#include "ptx.cuh"
#include "tile_order.h"

namespace edgelora {

struct TileCoord {
  int32_t row_r;     // first row of the W tile
  int32_t kb0, kb1;  // K blocks of this CTA's split
  int32_t split;
};

__device__ __forceinline__ TileCoord tile_coord(const GemmParams &p, int32_t bid) {
  TileCoord c;
  const int m = bid / p.splits;  // the splits of a row tile are consecutive CTAs: one cluster
  c.split = bid - m * p.splits;
  c.row_r = m * kTileM;
  c.kb0 = min(p.kb_total, c.split * p.kb_per);
  c.kb1 = min(p.kb_total, c.kb0 + p.kb_per);
  return c;
}

// decode: first W row of the tile this CTA works on
__device__ __forceinline__ int32_t tc_row0(const GemmParams &p, int32_t bid) {
  return bid / p.splits * kTileM;
}

__device__ __forceinline__ void named_bar_sync(int id, int threads) {
  __syncwarp();  // (bar.sync is the aligned form)
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void st_cluster_f32(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster_f32x4(uint32_t addr, float a, float b, float c, float d) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d)
               : "memory");
}

__device__ __forceinline__ int32_t ld_acquire_gpu(const int32_t *ptr) {
  int32_t v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(ptr) : "memory");
  return v;
}

// Bounded wait of one thread for the shrink teams' arrival counter.
__device__ __forceinline__ int wait_for_teams(const int32_t *counter, int32_t n, long long wl, uint32_t *status) {
  const long long t_start = clock64();
  while (ld_acquire_gpu(counter) < n) {
    if (clock64() - t_start > wl) {
      atomicOr(status, EDGELORA_STATUS_TIMEOUT);
      return 0;
    }
  }
  return 1;
}

// Fused decode launches (batches of at most 64 tokens): z[t] = s_a A_a x[t] on the CUDA cores, by
// "teams" of four warps: warps 6..9 of every CTA of the decode job and two teams in every spare CTA.
// A team item is (token, eight rank rows, K chunk): chunk c covers the K steps c, c + ks, ... of 256
// elements; warp w of the team takes every fourth of them, lane l the elements [8 l, 8 l + 8) of a
// step (one 16-byte load of x and eight of A in flight per lane).  The four warps' sums meet in
// shared memory and are added in a fixed order; the partial result goes to plane c of f.z, and the
// expand adds the planes in order.  Rows at or past the rank are never read by the expand and are
// not written.  s_tid / s_trank / s_tscale: the tokens' validated ids, ranks and scales in shared
// memory; s_red: 48 floats; bar_id: a named barrier of the team's 128 threads.
template <int kBarId>
__device__ __forceinline__ void shrink_team_items(const GemmParams &p, const FusedDecode &f, int team, int n_teams,
                                                  int wt, int lane, const int32_t *s_tid, const int32_t *s_trank,
                                                  const float *s_tscale, float *s_red, bool &waited) {
  const int n_ksteps = (p.h_in + kShrinkStepElems - 1) / kShrinkStepElems;
  const int n_rgn = p.R_pad >> 3, KS = f.ks;
  const int n_items = p.T * n_rgn * KS;
  const size_t zplane = static_cast<size_t>(p.max_tokens) * p.R_pad;
  const int row_u4 = p.h_in >> 3;  // 16-byte pieces of a row (h_in is a multiple of 8)
  int par = 0;
  for (int item = team; item < n_items; item += n_teams) {
    const int c = item % KS, tr = item / KS;
    const int t = tr / n_rgn, rg = tr - t * n_rgn;
    const int at = s_tid[t], rank = s_trank[t];
    if (at < 0) continue;
    if (rank <= 0) {
      if (wt == 0 && lane == 0 && c == 0 && rg == 0) atomicOr(p.status, EDGELORA_STATUS_SLOT_EMPTY);
      continue;
    }
    if (rg * 8 >= rank) continue;  // zero padding of the block
    const uint4 *Arow =
        reinterpret_cast<const uint4 *>(f.A_pool + (static_cast<size_t>(at) * p.R_pad + rg * 8) * p.h_in);
    const uint4 *xrow = reinterpret_cast<const uint4 *>(f.x + static_cast<size_t>(t) * p.h_in);
    float acc[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) acc[r] = 0.f;
    for (int s0 = c + KS * wt; s0 < n_ksteps; s0 += 4 * KS) {
      const int k0 = s0 * 32 + lane;
      if (k0 >= row_u4) continue;
      uint4 av[8];
      const uint4 xv = __ldcg(xrow + k0);
#pragma unroll
      for (int r = 0; r < 8; ++r) av[r] = __ldg(Arow + static_cast<size_t>(r) * row_u4 + k0);
      const float xf[8] = {ptx::bf16_lo(xv.x), ptx::bf16_hi(xv.x), ptx::bf16_lo(xv.y), ptx::bf16_hi(xv.y),
                           ptx::bf16_lo(xv.z), ptx::bf16_hi(xv.z), ptx::bf16_lo(xv.w), ptx::bf16_hi(xv.w)};
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        float v = acc[r];
        v = fmaf(ptx::bf16_lo(av[r].x), xf[0], v);
        v = fmaf(ptx::bf16_hi(av[r].x), xf[1], v);
        v = fmaf(ptx::bf16_lo(av[r].y), xf[2], v);
        v = fmaf(ptx::bf16_hi(av[r].y), xf[3], v);
        v = fmaf(ptx::bf16_lo(av[r].z), xf[4], v);
        v = fmaf(ptx::bf16_hi(av[r].z), xf[5], v);
        v = fmaf(ptx::bf16_lo(av[r].w), xf[6], v);
        v = fmaf(ptx::bf16_hi(av[r].w), xf[7], v);
        acc[r] = v;
      }
    }
    float out = 0.f;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      float v = acc[r];
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
      if (lane == r) out = v;
    }
    // buffer `par` is written again two items later, behind the next item's barrier, which warp 0
    // reaches only after it has read this item's sums
    if (wt > 0 && lane < 8) s_red[(par * 3 + wt - 1) * 8 + lane] = out;
    named_bar_sync(kBarId, 128);
    if (wt == 0) {
      if (!waited) {  // first write of this team to memory that earlier kernels may read
        ptx::pdl_wait_prior_grids();
        waited = true;
      }
      if (lane < 8) {
        const float sum = ((out + s_red[(par * 3 + 0) * 8 + lane]) + s_red[(par * 3 + 1) * 8 + lane]) +
                          s_red[(par * 3 + 2) * 8 + lane];
        f.z[c * zplane + static_cast<size_t>(t) * p.R_pad + rg * 8 + lane] = s_tscale[t] * sum;
      }
    }
    par ^= 1;
  }
  if (wt == 0) {
    __syncwarp();  // the lanes' z stores happen before lane 0's release
    if (lane == 0) {
      ptx::pdl_wait_prior_grids();  // the counters belong to the kernel before this one until it is done
      __threadfence();
      atomicAdd(f.sync, 1);
    }
  }
}

// A spare CTA of a fused decode launch: two shrink teams (warps 0..3 and 4..7); the first spare CTA
// also publishes the routing plan.
__device__ __forceinline__ void fused_shrink_cta(const GemmParams &p, const FusedDecode &f, uint8_t *smem, int n_teams) {
  int32_t *s_id = reinterpret_cast<int32_t *>(smem);  // [256] validated ids
  int32_t *s_cnt = s_id + 256;                        // [256] scratch of the plan publication
  int32_t *s_rank = s_cnt + 256;                      // [256]
  float *s_scale = reinterpret_cast<float *>(s_rank + 256);  // [256]
  float *s_red = s_scale + 256;                              // [2][48]
  int *s_wt = reinterpret_cast<int *>(s_red + 96);           // [9]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  ptx::pdl_launch_dependents();
  int a = -1;
  bool bad = false;
  if (tid < p.T) {
    a = p.ids[tid];
    if (a < -1 || a >= p.n_slots) {
      a = -1;
      bad = true;
    }
  }
  SlotRow row = {0, 0.f, 0, 0};
  if (a >= 0) row = p.slots[a];
  if (tid < 256) {
    s_id[tid] = a;
    s_rank[tid] = row.rank;
    s_scale[tid] = row.scale;
  }
  const int any_bad = __syncthreads_or(bad ? 1 : 0);
  bool waited = false;
  if (f.x_wait) {
    ptx::pdl_wait_prior_grids();
    waited = true;
  }
  if (warp < 4)
    shrink_team_items<2>(p, f, static_cast<int>(blockIdx.x) * 2, n_teams, warp, lane, s_id, s_rank, s_scale, s_red,
                         waited);
  else if (warp < 8)
    shrink_team_items<3>(p, f, static_cast<int>(blockIdx.x) * 2 + 1, n_teams, warp - 4, lane, s_id, s_rank, s_scale,
                         s_red + 48, waited);
  if (blockIdx.x == 0) publish_decode_plan(f.pv, a, p.T, any_bad, f.ks, s_id, s_cnt, s_wt);
}

// kFused: a launch whose first f.n_ctas CTAs are shrink CTAs (fused_shrink_cta); the job's own CTAs are
// numbered from there.  Without it the registers are capped so that the CTAs fit beside the shrink kernel's.
template <bool kFused>
__global__ void __launch_bounds__(kGemmThreads, kFused ? 1 : 2)
lora_gemm_kernel(const __grid_constant__ CUtensorMap tmap_r, const __grid_constant__ CUtensorMap tmap_c,
                 const __grid_constant__ CUtensorMap tmap_b, const GemmParams p, const FusedDecode f) {
  extern __shared__ uint8_t smem_raw[];
  // tiles need 1024-byte alignment for the 128-byte swizzle
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int32_t cta0 = kFused ? f.n_ctas : 0;  // whole clusters: the cluster ranks of the others are unchanged
  const int32_t ngrid = static_cast<int32_t>(gridDim.x) - cta0;
  if (kFused && static_cast<int32_t>(blockIdx.x) < cta0) {
    fused_shrink_cta(p, f, smem, 2 * cta0 + ngrid);
    return;
  }
  const int32_t bid = static_cast<int32_t>(blockIdx.x) - cta0;
  const uint32_t r_bytes = kTileM * kBlockK * 2;              // 16 KB
  const uint32_t c_bytes = static_cast<uint32_t>(p.BN) * kBlockK * 2;
  const uint32_t stage_bytes = r_bytes + c_bytes;
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + static_cast<size_t>(p.stages) * stage_bytes);
  uint64_t *full_bar = bars;                      // [stages]  TMA -> MMA
  uint64_t *empty_bar = bars + kMaxStages;        // [stages]  MMA -> TMA
  uint64_t *tfull_bar = bars + 2 * kMaxStages;    //           MMA -> epilogue
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(tfull_bar + 4);
  volatile uint32_t *abort_flag = tmem_slot + 1;
  // 512 bytes after the barriers: what the owner of some tokens keeps of them, scratch of the shrink team
  uint8_t *extra = reinterpret_cast<uint8_t *>(bars) + 512;
  int32_t *s_rank = reinterpret_cast<int32_t *>(extra + 128);               // [16] of each of this CTA's tokens
  int32_t *s_vid = reinterpret_cast<int32_t *>(extra + 1152);               // [16] adapters, -1: none
  uint32_t *s_team = reinterpret_cast<uint32_t *>(extra + 2432);            // [256]
  volatile int32_t *s_last = reinterpret_cast<volatile int32_t *>(extra + 80);  // the wait for the shrink teams ended in time
  uint64_t *ep_bar = reinterpret_cast<uint64_t *>(extra + 88);              // the staged B_a rows have landed
  uint8_t *b_stage = reinterpret_cast<uint8_t *>(bars) + 4096;  // fused decode: B_a rows of the owner's tokens, then their z

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long wl = p.wait_cycles;  // limit of every bounded wait below
  const TileCoord tc = tile_coord(p, bid);

  if (threadIdx.x == 0) {
    ptx::prefetch_tensormap(&tmap_r);
    ptx::prefetch_tensormap(&tmap_c);
    for (int s = 0; s < p.stages; ++s) {
      ptx::mbar_init(&full_bar[s], 1);
      ptx::mbar_init(&empty_bar[s], 1);
    }
    ptx::mbar_init(tfull_bar, 1);
    ptx::mbar_init(ep_bar, 4);  // one arrival per epilogue warp
    *abort_flag = 0;
    ptx::fence_barrier_init();
    if (kFused && f.x_wait) {
      // W is not written by any kernel of this library: this thread (lane 0 of the producer warp, which
      // has just initialised the barriers) requests the W tiles of the first ring revolution at once,
      // before the tensor-memory allocation and the CTA-wide barrier; the producer adds the x tiles
      // after its dependency wait
      const int32_t npre = min(p.stages, tc.kb1 - tc.kb0);
      for (int32_t i = 0; i < npre; ++i) {
        ptx::mbar_arrive_expect_tx(&full_bar[i], r_bytes + c_bytes);
        ptx::tma_load_2d(smem + static_cast<size_t>(i) * stage_bytes, &tmap_r, &full_bar[i], (tc.kb0 + i) * kBlockK,
                         tc.row_r);
      }
    }
  }
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, static_cast<uint32_t>(p.tmem_cols));
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  // Every CTA of this grid now holds its tensor memory, so a dependent grid may start to launch.
  ptx::pdl_launch_dependents();

  const uint32_t nstages = static_cast<uint32_t>(p.stages);
  bool fused_z_ok = true;  // fused launches: set by the epilogue warps' wait for the shrink teams
  // (The issuing roles run behind elect.sync, not lane == 0: the compiler then knows that one thread issues, and
  // the tensor and TMA instructions, which take their operands from uniform registers, need no loop over the lanes.)
  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (ptx::elect_one()) {
      uint32_t stage = 0, phase = 0, used = 0;
      bool ok = true;
      auto wait_empty = [&]() { return ptx::mbar_wait(&empty_bar[stage], phase ^ 1, wl) && !*abort_flag; };
      auto advance = [&]() {
        ++used;
        if (++stage == nstages) {
          stage = 0;
          phase ^= 1;
        }
      };
      int32_t kb_first = tc.kb0;
      if (kFused && f.x_wait) {
        // x may be an output of the kernel before this one, W is not: the W tiles of the first ring
        // revolution were requested in the prologue (with the bytes of both tiles announced), the x
        // tiles follow the dependency wait
        const int32_t npre = min(static_cast<int32_t>(nstages), tc.kb1 - tc.kb0);  // the ring is empty: no waits
        ptx::pdl_wait_prior_grids();
        for (int32_t i = 0; i < npre; ++i) {
          ptx::tma_load_2d(smem + static_cast<size_t>(i) * stage_bytes + r_bytes, &tmap_c, &full_bar[i],
                           (tc.kb0 + i) * kBlockK, 0);
          advance();
        }
        kb_first += npre;
      }
      for (int32_t kb = kb_first; kb < tc.kb1; ++kb) {
        if (!wait_empty()) {
          ok = false;
          break;
        }
        uint8_t *sr = smem + static_cast<size_t>(stage) * stage_bytes;
        ptx::mbar_arrive_expect_tx(&full_bar[stage], r_bytes + c_bytes);
        ptx::tma_load_2d(sr, &tmap_r, &full_bar[stage], kb * kBlockK, tc.row_r);
        ptx::tma_load_2d(sr + r_bytes, &tmap_c, &full_bar[stage], kb * kBlockK, 0);
        advance();
      }
      if (!ok) {
        *abort_flag = 1;
        atomicOr(p.status, EDGELORA_STATUS_TIMEOUT);
      }
      // What was requested lands before the CTA frees its memory, also when a wait of some role ran out.
      const RingPos last = ring_drain(used, nstages);
      stage = last.stage;
      phase = last.phase;
      for (uint32_t i = min(used, nstages); i > 0; --i) {
        ptx::mbar_wait(&full_bar[stage], phase ^ 1);
        advance();
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (ptx::elect_one()) {
      const uint32_t idesc = ptx::umma_idesc_bf16(kTileM, static_cast<uint32_t>(p.BN));
      uint32_t stage = 0, phase = 0;
      bool ok = true;
      for (int32_t kb = tc.kb0; kb < tc.kb1; ++kb) {
        if (!ptx::mbar_wait(&full_bar[stage], phase, wl) || *abort_flag) {
          ok = false;
          break;
        }
        ptx::tc_fence_after_sync();
        const uint32_t sr = ptx::smem_u32(smem + static_cast<size_t>(stage) * stage_bytes);
        const uint64_t da = ptx::umma_desc_k128(sr);
        const uint64_t db = ptx::umma_desc_k128(sr + r_bytes);
#pragma unroll
        for (int k = 0; k < kBlockK / kUmmaK; ++k) {
          // advancing 16 bf16 along K inside the swizzled row = 32 bytes = 2 descriptor units
          ptx::umma_bf16(tmem_base, da + 2 * k, db + 2 * k, idesc, (kb > tc.kb0 || k > 0) ? 1u : 0u);
        }
        ptx::umma_commit(&empty_bar[stage]);  // frees the smem stage once these MMAs are done
        if (++stage == nstages) {
          stage = 0;
          phase ^= 1;
        }
      }
      if (!ok) {
        *abort_flag = 1;
        atomicOr(p.status, EDGELORA_STATUS_TIMEOUT);
      }
      ptx::umma_commit(tfull_bar);  // accumulator complete, or as far as it came (the flag says which)
      ptx::mbar_wait(tfull_bar, 0);  // this warp frees the tensor memory: nothing writes to it any more

    }
  } else if (warp < 6) {
    // ------------------------------------------------------------ epilogue (warps 2..5)
    const int quad = warp & 3;  // TMEM lanes [32*quad, 32*quad+32)
    if (kFused && f.b_stage) {
      // This CTA will finish tokens [rank * cols_per, ...) of its row tile: the B_a rows they need (the
      // tile's 128 rows of the token's adapter) are copied into shared memory now, one copy per token, while the main
      // loop runs (the ids are the caller's input, the pool is not written by this kernel).  One warp per token;
      // cols_per <= 16.
      const int cols_per = p.BN / p.splits;
      const int t0 = static_cast<int>(ptx::cluster_rank()) * cols_per;
      const uint32_t tok_bytes = kTileM * p.R_pad * 2;
      int32_t a_of[4];
      uint32_t my_bytes = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int cl = quad + 4 * i;
        int32_t a = -1, rank = 0;
        if (cl < cols_per && t0 + cl < p.T) {
          a = p.ids[t0 + cl];
          if (a < 0 || a >= p.n_slots) a = -1;
          if (a >= 0) rank = p.slots[a].rank;
        }
        if (rank <= 0) a = -1;
        a_of[i] = a;
        if (cl < cols_per && lane == 0) {  // kept for the expand at the end
          s_vid[cl] = a;
          s_rank[cl] = rank;
        }
        if (a >= 0) my_bytes += tok_bytes;
      }
      if (lane == 0) {
        ptx::mbar_arrive_expect_tx(ep_bar, my_bytes);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (a_of[i] >= 0)
            ptx::tma_load_3d(b_stage + static_cast<size_t>(quad + 4 * i) * tok_bytes, &tmap_b, ep_bar, 0, tc_row0(p, bid),
                             a_of[i]);
      }
    } else {
      // This CTA will finish tokens [rank * cols_per, ...) of its row tile; pull the B_a rows they
      // need into L2 now (the ids are the caller's input, the pool is not written by the shrink).
      const int cols_per = p.BN / p.splits;
      const int t0 = static_cast<int>(ptx::cluster_rank()) * cols_per;
      for (int cl = quad; cl < cols_per; cl += 4) {  // one warp per token
        int32_t a = -1, rank = 0;
        if (t0 + cl < p.T) {
          a = p.ids[t0 + cl];
          if (a < 0 || a >= p.n_slots) a = -1;
          if (a >= 0) rank = p.slots[a].rank;
        }
        if (lane == 0) {  // kept for the expand at the end
          s_vid[cl] = rank > 0 ? a : -1;
          s_rank[cl] = rank;
        }
        if (t0 + cl < p.T) {
          if (a >= 0 && a < p.n_slots) {
            const uint8_t *rows = reinterpret_cast<const uint8_t *>(
                p.B_pool + (static_cast<size_t>(a) * p.h_out + tc_row0(p, bid)) * p.R_pad);
            const int bytes = min(kTileM, p.h_out - tc_row0(p, bid)) * p.R_pad * 2;  // this tile's rows, contiguous
            for (int off = lane * 128; off < bytes; off += 32 * 128)
              asm volatile("prefetch.global.L2 [%0];" ::"l"(rows + off));
          }
        }
      }
    }
    if (kFused && !f.b_stage) {
      // z comes from the shrink teams of this grid (every CTA of the launch is resident, so all of them run): bounded wait
      // for their arrival counter.  The counter belongs to the kernel before this one (another launch of this pool, which
      // leaves it at zero) until that kernel is done.
      ptx::pdl_wait_prior_grids();
      // one thread of the CTA polls; the named barrier of the four warps passes its acquire on
      if (warp == 2 && lane == 0) *s_last = wait_for_teams(f.sync, 2 * cta0 + ngrid, wl, p.status);
      named_bar_sync(1, 128);
      fused_z_ok = *s_last != 0;
    }
    const bool ok = ptx::mbar_wait(tfull_bar, 0, wl) && !*abort_flag;
    __syncwarp();
    if (!ok) {
      *abort_flag = 1;
      if (lane == 0) atomicOr(p.status, EDGELORA_STATUS_TIMEOUT);
    }
  } else if (kFused) {
    // ------------------------------------------------------------ shrink team (warps 6..9)
    const int btid = threadIdx.x - 192;  // 0..127
    int32_t *s_tid = reinterpret_cast<int32_t *>(s_team) + 64;
    int32_t *s_trank = s_tid + 64;
    float *s_tscale = reinterpret_cast<float *>(s_trank + 64);
    if (btid < 64) {
      int32_t a = -1;
      if (btid < p.T) {
        a = p.ids[btid];
        if (a < 0 || a >= p.n_slots) a = -1;
      }
      SlotRow row = {0, 0.f, 0, 0};
      if (a >= 0) row = p.slots[a];
      s_tid[btid] = a;
      s_trank[btid] = row.rank;
      s_tscale[btid] = row.scale;
    }
    named_bar_sync(2, 128);
    bool waited = false;
    if (f.x_wait) {
      ptx::pdl_wait_prior_grids();
      waited = true;
    }
    shrink_team_items<2>(p, f, 2 * cta0 + bid, 2 * cta0 + ngrid, warp - 6, lane, s_tid, s_trank, s_tscale,
                         reinterpret_cast<float *>(s_team), waited);
  }

  {
    // ---------------------------------------------------------- split-K reduction in the cluster
    // CTA `rank` of the cluster owns tokens [rank * cols_per, (rank + 1) * cols_per).  Its buffer
    // buf[src split][token][row] overlays the operand ring, which is idle once every CTA of the
    // cluster is past its main loop (first barrier).
    const bool epi = warp >= 2 && warp < 6;
    const int quad = warp & 3, row_in_tile = quad * 32 + lane, etid = threadIdx.x - 64;
    const uint32_t my_rank = ptx::cluster_rank();
    const int cols_per = p.BN / p.splits;  // a power of two (BN and splits are)
    const int shift = 31 - __clz(cols_per);
    const bool have_acc = epi && !*abort_flag;  // this CTA's accumulator is complete (tfull waited)
    const bool z_ok = fused_z_ok;  // fused launches: the wait for the shrink teams ended in time
    float4 *z_stage = reinterpret_cast<float4 *>(b_stage + static_cast<size_t>(cols_per) * kTileM * p.R_pad * 2);
    // The partial tiles land in the operand ring, which is idle once every CTA of the cluster is past
    // its main loop: hence the first barrier.  A fused launch with room to spare (b_stage == 2) has a
    // buffer of its own behind the staged rows instead, and sends at once.
    const bool own_buf = kFused && f.b_stage == 2;
    uint8_t *red = own_buf ? b_stage + ((static_cast<size_t>(cols_per) * (kTileM * p.R_pad * 2 + p.R_pad * 4) + 1023) &
                                        ~static_cast<size_t>(1023))
                           : smem;
    __syncwarp();
    if (!own_buf) ptx::cluster_sync_all();
    if (have_acc) {
      ptx::tc_fence_after_sync();
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
      const uint32_t local = ptx::smem_u32(red) +
                             ((my_rank * cols_per) * kTileM + row_in_tile) * 4u;
      const uint32_t qpo = static_cast<uint32_t>(cols_per) >> 2;  // token quads per owner
      for (int32_t c0 = 0; c0 < p.BN; c0 += 32) {
        float v[32];
        ptx::tmem_ld_32x32(taddr + c0, v);
        if (!(kFused && f.b_stage)) {  // buf[src][token][row]
#pragma unroll
          for (int jj = 0; jj < 32; ++jj) {
            const int col = c0 + jj;
            const uint32_t owner = static_cast<uint32_t>(col >> shift);
            const uint32_t off = static_cast<uint32_t>(col & (cols_per - 1)) * kTileM * 4u;
            st_cluster_f32(ptx::map_to_rank(local + off, owner), v[jj]);  // a warp writes 128 bytes in a row
          }
        } else {  // buf[src][token quad][row][4 tokens]: 16-byte stores, a warp writes 512 bytes in a row
#pragma unroll
          for (int g4 = 0; g4 < 8; ++g4) {
            const int col = c0 + g4 * 4;
            const uint32_t owner = static_cast<uint32_t>(col >> shift);
            const uint32_t quad_i = static_cast<uint32_t>(col & (cols_per - 1)) >> 2;
            const uint32_t addr = ptx::smem_u32(red) + ((my_rank * qpo + quad_i) * kTileM + row_in_tile) * 16u;
            st_cluster_f32x4(ptx::map_to_rank(addr, owner), v[g4 * 4], v[g4 * 4 + 1], v[g4 * 4 + 2], v[g4 * 4 + 3]);
          }
        }
      }
    }
    __syncwarp();
    if (kFused && f.b_stage) {
      // Small batches, one launch.  The partial sums are on their way; while the cluster's other CTAs send theirs, the
      // epilogue and team warps (2..9) work out the expand of this CTA's tokens: z, which the team has brought to shared
      // memory, against the staged B_a rows, a thread per W row and every other token quad.
      // (With the expand behind the exchange, by the epilogue warps alone, the tail behind the last MMA took 6 us for 32
      // tokens and 9 for 64: 4096 -> 4096, 32 tokens 15.1 us per call, now 12.3; 64 tokens 18.0 and 14.1; 256 -> 256, 16
      // tokens 7.9 and 5.7.)
      ptx::cluster_arrive();
      const int half = warp >= 6 ? 1 : 0, nq = cols_per >> 2, R4 = p.R_pad >> 2;
      const int r = (threadIdx.x - 64) & 127;
      float e[2][4];
#pragma unroll
      for (int i = 0; i < 8; ++i) e[i >> 2][i & 3] = 0.f;
      int passed = 0;
      if (warp >= 6) {
        // Behind its items the team waits for the others and brings z of the tokens that this CTA will finish to shared memory,
        // the K chunks' planes added in order.  With a long K that is over before the accumulator is.  (By the epilogue warps, behind
        // it, and here, us per call: 8192 -> 512, one token on rank 32: 7.9 and 6.9; 14336 -> 1024, one token on rank 16: 11.4 and
        // 10.4; 4096 -> 4096, four tokens: 10.8 and 9.8, 32 tokens: 11.9 and 11.2; 2048 -> 2048, eight tokens: 7.1 and 6.2.)
        const int32_t *s_tid = reinterpret_cast<const int32_t *>(s_team) + 64, *s_trank = s_tid + 64;
        if (warp == 6) {
          // the counter belongs to the kernel before this one (another launch of this pool, which leaves it at zero) until
          // that kernel is done
          ptx::pdl_wait_prior_grids();
          // one thread of the CTA polls; the named barriers pass its acquire on
          if (lane == 0) *s_last = wait_for_teams(f.sync, 2 * cta0 + ngrid, wl, p.status);
        }
        named_bar_sync(2, 128);
        const bool in_time = *s_last != 0;
        const size_t zplane4 = static_cast<size_t>(p.max_tokens) * R4;
        for (int i = static_cast<int>(threadIdx.x) - 192; i < cols_per * R4; i += 128) {
          const int cl = i / R4, c4 = i - cl * R4, t = static_cast<int>(my_rank) * cols_per + cl, rank = s_trank[t];
          float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
          if (s_tid[t] >= 0 && rank > 0 && in_time) {
            const float4 *zp = reinterpret_cast<const float4 *>(f.z) + static_cast<size_t>(t) * R4 + c4;
            float4 w[8];
            for (int s0 = 0; s0 < f.ks; s0 += 8) {
#pragma unroll
              for (int k = 0; k < 8; ++k) w[k] = s0 + k < f.ks ? __ldcg(zp + (s0 + k) * zplane4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                z.x += w[k].x; z.y += w[k].y; z.z += w[k].z; z.w += w[k].w;
              }
            }
            // (what lies behind the last live group of eight rank rows was not written)
            if (c4 * 4 + 0 >= rank) z.x = 0.f;
            if (c4 * 4 + 1 >= rank) z.y = 0.f;
            if (c4 * 4 + 2 >= rank) z.z = 0.f;
            if (c4 * 4 + 3 >= rank) z.w = 0.f;
          }
          z_stage[i] = z;
        }
      }
      if (warp >= 2) {
        named_bar_sync(3, 256);  // z of this CTA's tokens is there
        // the wait for the shrink teams is over in this CTA (see the end)
        if (epi && lane == 0) passed = atomicAdd(f.sync + 1, 1);
        bool z_ok = *s_last != 0;
        if (!__all_sync(0xffffffffu, ptx::mbar_wait(ep_bar, 0, max(wl, ptx::kSettleCycles)))) {  // the staged B_a rows
          if (lane == 0) atomicOr(p.status, EDGELORA_STATUS_TIMEOUT);
          z_ok = false;
        }
        const int sw = row_swizzle(r, p.R_pad);
        const uint32_t brow = ptx::smem_u32(b_stage) + r * p.R_pad * 2, tok_bytes = kTileM * p.R_pad * 2;
        const uint32_t zrow = ptx::smem_u32(z_stage);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int qd = half + 2 * i;
          if (qd < nq) {
            uint32_t live[4];
            uint64_t s0[4], s1[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              live[k] = z_ok && s_vid[qd * 4 + k] >= 0 ? 1u : 0u;
              s0[k] = s1[k] = 0;
            }
#pragma unroll 2
            for (int c = 0; c < p.R_pad / 8; ++c) {
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const int cl = qd * 4 + k;
                uint64_t b0, b1, u[4];
                ptx::ld_shared_f32x4_if(brow + cl * tok_bytes + ((c ^ sw) << 4), live[k], b0, b1);
                ptx::ld_shared_f32x4_if(zrow + (cl * R4 + 2 * c) * 16, 1u, u[0], u[1]);
                ptx::ld_shared_f32x4_if(zrow + (cl * R4 + 2 * c + 1) * 16, 1u, u[2], u[3]);
                const uint32_t w0 = static_cast<uint32_t>(b0), w1 = static_cast<uint32_t>(b0 >> 32);
                const uint32_t w2 = static_cast<uint32_t>(b1), w3 = static_cast<uint32_t>(b1 >> 32);
                s0[k] = ptx::fma_f32x2(ptx::f32x2(ptx::bf16_lo(w0), ptx::bf16_hi(w0)), u[0], s0[k]);
                s1[k] = ptx::fma_f32x2(ptx::f32x2(ptx::bf16_lo(w1), ptx::bf16_hi(w1)), u[1], s1[k]);
                s0[k] = ptx::fma_f32x2(ptx::f32x2(ptx::bf16_lo(w2), ptx::bf16_hi(w2)), u[2], s0[k]);
                s1[k] = ptx::fma_f32x2(ptx::f32x2(ptx::bf16_lo(w3), ptx::bf16_hi(w3)), u[3], s1[k]);
              }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) e[i][k] = ptx::sum_f32x2(s0[k], s1[k]);
          }
        }
      }
      ptx::cluster_wait();
      if (warp >= 2) {
        const float4 *buf4 = reinterpret_cast<const float4 *>(red);
        const int j = bid / p.splits * kTileM + r;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int qd = half + 2 * i, t0 = static_cast<int>(my_rank) * cols_per + qd * 4;
          if (qd < nq && j < p.h_out) {
            float4 a4 = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
            for (int sp = 0; sp < p.splits; ++sp) {
              const float4 w = buf4[(sp * nq + qd) * kTileM + r];
              a4.x += w.x; a4.y += w.y; a4.z += w.z; a4.w += w.w;
            }
            const float o[4] = {a4.x + e[i][0], a4.y + e[i][1], a4.z + e[i][2], a4.w + e[i][3]};
#pragma unroll
            for (int k = 0; k < 4; ++k)
              if (t0 + k < p.T)
                p.y[static_cast<size_t>(t0 + k) * p.h_out + j] = static_cast<uint16_t>(ptx::pack_bf16x2(o[k], 0.f) & 0xFFFFu);
          }
        }
        // the last epilogue warp of the grid to pass its wait puts both counters back to zero for the next launch
        if (epi && lane == 0 && passed == ngrid * 4 - 1) {
          f.sync[0] = 0;
          f.sync[1] = 0;
        }
      }
    } else {
      ptx::cluster_sync_all();
      if (epi) {
        const float *buf = reinterpret_cast<const float *>(red);
        const int n_units = cols_per * 32;  // unit = (token, 4 adjacent W rows)
        const int row0 = bid / p.splits * kTileM;
        auto sum_partials = [&](int cl, int r4) {
          float4 acc4 = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int sp = 0; sp < p.splits; ++sp) {
            const float4 w = *reinterpret_cast<const float4 *>(buf + ((sp * cols_per + cl) * kTileM + r4));
            acc4.x += w.x; acc4.y += w.y; acc4.z += w.z; acc4.w += w.w;
          }
          return acc4;
        };
        auto store4 = [&](int t, int j, const float4 &v) {
          uint2 o;
          o.x = ptx::pack_bf16x2(v.x, v.y);
          o.y = ptx::pack_bf16x2(v.z, v.w);
          *reinterpret_cast<uint2 *>(p.y + static_cast<size_t>(t) * p.h_out + j) = o;
        };
        {
          // Small batches: wait for the shrink kernel (and for earlier readers of y), then per unit add the
          // splits' partial sums, fetch z and the B_a rows in one round trip, add B_a[j..j+3][0..r) . z[t]
          // in fp32 (z carries s_a) and write y.  A rolled loop over the units (at most 4 per thread:
          // cols_per <= 16): this code runs once per launch, and what it costs is mostly the fetching
          // of its instructions.
          ptx::pdl_wait_prior_grids();
          const int nch = p.R_pad >> 3;
          const int n_zp = kFused ? f.ks : 1;
          const size_t zplane4 = static_cast<size_t>(p.max_tokens) * p.R_pad / 4;
          auto load_z4 = [&](const float4 *ptr) {
            float4 v = __ldcg(ptr);
            for (int sp = 1; sp < n_zp; ++sp) {
              const float4 w = __ldcg(ptr + sp * zplane4);
              v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
            }
            return v;
          };
#pragma unroll 1
          for (int u = etid; u < n_units; u += 128) {
            const int cl = u >> 5, r4 = (u & 31) << 2;
            const int t = static_cast<int>(my_rank) * cols_per + cl, j = row0 + r4;
            if (t >= p.T || j >= p.h_out) continue;
            float4 acc4 = sum_partials(cl, r4);
            const int32_t a = z_ok ? s_vid[cl] : -1, rank = s_rank[cl];  // stored by the epilogue warps at the start
            if (a >= 0) {
              const uint4 *Brow = reinterpret_cast<const uint4 *>(
                  p.B_pool + (static_cast<size_t>(a) * p.h_out + j) * p.R_pad);
              const float4 *zt = reinterpret_cast<const float4 *>((kFused ? f.z : p.zws) + static_cast<size_t>(t) * p.R_pad);
              float add[4] = {0.f, 0.f, 0.f, 0.f};
              for (int c0 = 0; c0 < nch && c0 * 8 < rank; c0 += 2) {
                uint4 b[2][4];
                float4 z4[2][2];
#pragma unroll
                for (int cc = 0; cc < 2; ++cc) {  // two chunks of 8 rank values: 12 loads in flight
                  const int c = c0 + cc;
                  const bool on = c < nch && c * 8 < rank;
#pragma unroll
                  for (int r = 0; r < 4; ++r) b[cc][r] = on ? __ldg(Brow + r * nch + c) : make_uint4(0u, 0u, 0u, 0u);
                  z4[cc][0] = on ? load_z4(zt + 2 * c) : make_float4(0.f, 0.f, 0.f, 0.f);
                  z4[cc][1] = on ? load_z4(zt + 2 * c + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int cc = 0; cc < 2; ++cc) {
                  const float4 u0 = z4[cc][0], u1 = z4[cc][1];
#pragma unroll
                  for (int r = 0; r < 4; ++r) {
                    const uint4 bb = b[cc][r];
                    float s4 = add[r];
                    s4 = fmaf(ptx::bf16_lo(bb.x), u0.x, s4);
                    s4 = fmaf(ptx::bf16_hi(bb.x), u0.y, s4);
                    s4 = fmaf(ptx::bf16_lo(bb.y), u0.z, s4);
                    s4 = fmaf(ptx::bf16_hi(bb.y), u0.w, s4);
                    s4 = fmaf(ptx::bf16_lo(bb.z), u1.x, s4);
                    s4 = fmaf(ptx::bf16_hi(bb.z), u1.y, s4);
                    s4 = fmaf(ptx::bf16_lo(bb.w), u1.z, s4);
                    s4 = fmaf(ptx::bf16_hi(bb.w), u1.w, s4);
                    add[r] = s4;
                  }
                }
              }
              acc4.x += add[0]; acc4.y += add[1]; acc4.z += add[2]; acc4.w += add[3];
            }
            store4(t, j, acc4);
          }
          if (kFused && lane == 0) {
            // this warp is past its wait for the shrink teams: the last such warp of the grid puts both
            // counters back to zero for the next launch
            if (atomicAdd(f.sync + 1, 1) == ngrid * 4 - 1) {
              f.sync[0] = 0;
              f.sync[1] = 0;
            }
          }
        }
      }
    }
  }

  ptx::tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tmem_base, static_cast<uint32_t>(p.tmem_cols));
  }
}

cudaError_t gemm_set_smem_limit(size_t smem_bytes) {
  cudaError_t e = cudaSuccess;
  const int bytes = static_cast<int>(smem_bytes);
#define EDGELORA_SMEM(FU)                                                                                       \
  if (e == cudaSuccess)                                                                                     \
    e = cudaFuncSetAttribute(lora_gemm_kernel<FU>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  EDGELORA_SMEM(false)
  EDGELORA_SMEM(true)
#undef EDGELORA_SMEM
  return e;
}

cudaError_t launch_gemm(const CUtensorMap &tmap_row, const CUtensorMap &tmap_col, const GemmParams &p, int32_t grid,
                        size_t smem_bytes, bool pdl, cudaStream_t stream) {
  return launch_ex(lora_gemm_kernel<false>, dim3(grid), dim3(kGemmThreads), smem_bytes, stream, pdl, p.splits, tmap_row, tmap_col,
                   tmap_row, p, FusedDecode{});
}

cudaError_t launch_gemm_fused(const CUtensorMap &tmap_row, const CUtensorMap &tmap_col, const CUtensorMap &tmap_b, const GemmParams &p,
                              const FusedDecode &f, size_t smem_bytes, bool pdl, cudaStream_t stream) {
  const int32_t grid = f.n_ctas + p.n_mtiles * p.splits;
  return launch_ex(lora_gemm_kernel<true>, dim3(grid), dim3(kGemmThreads), smem_bytes, stream, pdl, p.splits,
                   tmap_row, tmap_col, tmap_b, p, f);
}

int32_t gemm_fused_max_ctas(int32_t cluster, size_t smem_bytes) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(cluster) * 64);
  cfg.blockDim = dim3(kGemmThreads);
  cfg.dynamicSmemBytes = smem_bytes;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(cluster);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, lora_gemm_kernel<true>, &cfg);
  if (getenv("EDGELORA_LOG"))
    fprintf(stderr, "edgelora: one-launch decode, clusters of %d, %zu bytes of shared memory: %s, %d clusters fit\n",
            cluster, smem_bytes, cudaGetErrorString(e), n);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n * cluster;
}

}  // namespace edgelora
