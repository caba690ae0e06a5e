// Base product and expand of one linear site over a decode-sized batch (paper Section 3.4), for the batches that the
// one-launch path of gemm.cu does not take: more than 64 tokens, or too many for the row tiles that the site has.
//
// D[128 x N] (fp32, in tensor memory) = R[128 x K] * C[N x K]^T, R = 128 rows of W, C = all tokens, K blocks of 64 from a TMA
// ring, K split over the `parts` CTAs of a cluster.  Each CTA finishes some tokens of the tile: it gets the other parts' sums
// of their columns through distributed shared memory, and works out their expand itself, on the CUDA cores from fp32 z,
// beside the stream of W: the B_a rows of its tokens' adapters and the tokens' z rows come through a ring of their own.
// Neither the K blocks nor the exchange wait for z, an adapter's values reach its own tokens' rows only, and a CTA looks at
// its own tokens' ids only.  Figures: see decode_parts in pool.cu.
//
// Warp roles: warp 0 issues the loads of W and x (the first round of the ring before anything else), warp 1 owns tensor memory
// and issues the MMAs, warps 2 and 3 issue the copies of the expand, each those of one of the two groups of expand warps,
// warps 4..11 (two to a lane quadrant: a single warp per scheduler cannot keep up with the latency of its sums) work out the
// u-batches, the expand and y.  (A thread takes 0.3 us to issue the copies of a stage; with all stages issued by one warp that
// was the pace of an expand of rank stride 16 or 32: 336 -> 13208, 209 tokens on 17 adapters: 37.1 us per call, now 31.7; 512 ->
// 11744, 119 tokens on 25, A in Q8_0: 28.9 and 25.5; 1848 -> 288, 255 tokens on 56: 36.0 and 34.4.  At stride 64 the reads of
// z and B from shared memory are.)  Every mbarrier wait is bounded; on a
// timeout the status word gets EDGELORA_STATUS_TIMEOUT and all roles leave.
#include <algorithm>

#include "decode_route.cuh"
#include "decode_tile.h"
#include "expand.cuh"
#include "launch.cuh"
#include "ptx.cuh"

namespace edgelora {

namespace {

constexpr int kThreads = 384, kExpandThreads = 256;
// Stages of the expand's ring.  Even: the two groups of warps take alternate stages, and a group may wait for the second use of
// a ring position only if it was the one that saw the first (a wait for the phase behind one that is not over passes at once).
constexpr int kExpStages = 4;
static_assert(kExpStages % 2 == 0, "positions alternate between the groups");
constexpr uint32_t kWBytes = kTileM * kBlockK * 2;
constexpr size_t kTailBytes = 8192;

// What the rings may take; the exchange of the parts takes the same memory afterwards.
constexpr size_t kRingBytes = kTileSmemBudget - 1024 - kTailBytes;

struct Shared {
  uint64_t full[kTileMaxStages];       // TMA -> MMA
  uint64_t empty[kTileMaxStages];      // MMA -> TMA
  uint64_t bfull[kExpStages];   // copies of the expand -> expand warps
  uint64_t bempty[kExpStages];  // expand warps -> copies of the expand
  uint64_t tfull;                      // MMA -> expand warps
  uint64_t groups_ready;               // expand warps -> copies of the expand
  uint64_t parts;                      // the other parts of this CTA's columns have arrived
  uint32_t tmem_slot;
  volatile uint32_t abort_flag;
  uint8_t rank[kDecodeMaxT];           // of every group's adapter
  Groups groups;
};
static_assert(sizeof(Shared) <= kTailBytes, "tail of the shared memory");

// Rank, tokens and first position of an expand stage, in one word.
__device__ __forceinline__ uint32_t stage_info(const Shared &sh, int s) {
  const int g = sh.groups.block_group[s], pos = sh.groups.block_pos[s];
  return sh.rank[g] | min(kExpTok, sh.groups.start[g + 1] - pos) << 8 | pos << 16;
}

// The stage's tokens, four, two or one at a time, each into its column.
template <int kChunks>
__device__ __forceinline__ void expand_stage(const uint8_t *brow, int sw, uint32_t z, uint32_t z_bytes, int rank, int nt,
                                             uint32_t texp, const uint8_t *columns) {
  float acc[4];
#pragma unroll 1
  for (; nt >= 4; nt -= 4, z += 4 * z_bytes, columns += 4) {
    expand_dots<kChunks, 4>(brow, sw, z, z_bytes, rank, acc);
#pragma unroll
    for (int q = 0; q < 4; ++q) ptx::tmem_st_32x1(texp + columns[q], &acc[q]);
  }
  if (nt & 2) {
    expand_dots<kChunks, 2>(brow, sw, z, z_bytes, rank, acc);
    ptx::tmem_st_32x1(texp + columns[0], &acc[0]);
    ptx::tmem_st_32x1(texp + columns[1], &acc[1]);
    z += 2 * z_bytes;
    columns += 2;
  }
  if (nt & 1) {
    expand_dots<kChunks, 1>(brow, sw, z, z_bytes, rank, acc);
    ptx::tmem_st_32x1(texp + columns[0], &acc[0]);
  }
}

}  // namespace

__global__ void __launch_bounds__(kThreads, 1) decode_tile_kernel(const __grid_constant__ DecTile p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t stage_bytes = kWBytes + static_cast<uint32_t>(p.N) * (kBlockK * 2);
  const uint32_t nstages = static_cast<uint32_t>(p.stages), nexp = kExpStages;
  uint8_t *exp_ring = smem + static_cast<size_t>(nstages) * stage_bytes;
  Shared &sh = *reinterpret_cast<Shared *>(smem + kRingBytes);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long wl = p.wait_cycles;
  const int32_t tile = static_cast<int32_t>(blockIdx.x) / p.parts, part = static_cast<int32_t>(blockIdx.x) - tile * p.parts;
  const int32_t row0 = tile * kTileM, kb0 = part * p.kb / p.parts, kb1 = (part + 1) * p.kb / p.parts;
  // token quads, those of an owner, and this CTA's: its tokens are [t0, t0 + n_own)
  const int32_t n_quads = (p.T + 3) >> 2, per = (n_quads + p.parts - 1) / p.parts;
  const int32_t q0 = part * per, nq = max(0, min(per, n_quads - q0)), t0 = q0 * 4, n_own = max(0, min(nq * 4, p.T - t0));
  auto load_stage = [&](int32_t kb, uint32_t stage) {
    uint8_t *sr = smem + static_cast<size_t>(stage) * stage_bytes;
    ptx::mbar_arrive_expect_tx(&sh.full[stage], stage_bytes);
    ptx::tma_load_2d(sr, &p.w, &sh.full[stage], kb * kBlockK, row0);
    ptx::tma_load_2d(sr + kWBytes, &p.x, &sh.full[stage], kb * kBlockK, 0);
  };

  if (tid == 0) {
    for (uint32_t s = 0; s < nstages; ++s) {
      ptx::mbar_init(&sh.full[s], 1);
      ptx::mbar_init(&sh.empty[s], 1);
    }
    for (uint32_t s = 0; s < nexp; ++s) {
      ptx::mbar_init(&sh.bfull[s], 1);
      ptx::mbar_init(&sh.bempty[s], 4);  // one arrival per warp of the group that takes the stage
    }
    ptx::mbar_init(&sh.tfull, 1);
    ptx::mbar_init(&sh.groups_ready, 1);
    ptx::mbar_init(&sh.parts, 1);
    sh.abort_flag = 0;
    ptx::fence_barrier_init();
    // W and x are not written by the kernel in front of this one
    for (int32_t i = 0; i < min(kb1 - kb0, p.stages); ++i) load_stage(kb0 + i, i);
  }
  if (warp == 1) {
    ptx::tmem_alloc(&sh.tmem_slot, static_cast<uint32_t>(p.tmem_cols));
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  ptx::pdl_launch_dependents();
  const uint32_t tmem_acc = sh.tmem_slot, tmem_exp = tmem_acc + static_cast<uint32_t>((p.N + 31) & ~31);
  bool ok = true;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (W and x)
    if (ptx::elect_one()) {
      uint32_t stage = 0, phase = 1;
      for (int32_t kb = kb0 + p.stages; kb < kb1; ++kb) {
        if (!ptx::mbar_wait(&sh.empty[stage], phase ^ 1, wl) || sh.abort_flag) {
          ok = false;
          break;
        }
        load_stage(kb, stage);
        if (++stage == nstages) {
          stage = 0;
          phase ^= 1;
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (ptx::elect_one()) {
      const uint32_t idesc = ptx::umma_idesc_bf16(kTileM, static_cast<uint32_t>(p.N));
      uint32_t stage = 0, phase = 0;
      for (int32_t kb = kb0; kb < kb1; ++kb) {
        if (!ptx::mbar_wait(&sh.full[stage], phase, wl) || sh.abort_flag) {
          ok = false;
          break;
        }
        ptx::tc_fence_after_sync();
        const uint32_t sr = ptx::smem_u32(smem + static_cast<size_t>(stage) * stage_bytes);
        const uint64_t da = ptx::umma_desc_k128(sr), db = ptx::umma_desc_k128(sr + kWBytes);
#pragma unroll
        for (int k = 0; k < kBlockK / kUmmaK; ++k)
          ptx::umma_bf16(tmem_acc, da + 2 * k, db + 2 * k, idesc, (kb > kb0 || k > 0) ? 1u : 0u);
        ptx::umma_commit(&sh.empty[stage]);
        if (++stage == nstages) {
          stage = 0;
          phase ^= 1;
        }
      }
      ptx::umma_commit(&sh.tfull);  // accumulator complete, or as far as it came
    }
  } else if (warp < 4) {
    // ------------------------------------------------------------ copies of the expand (B_a rows and z; warps 2 and 3)
    const int half = warp - 2;
    ok = __all_sync(0xffffffffu, ptx::mbar_wait(&sh.groups_ready, 0, wl));
    ptx::pdl_wait_prior_grids();  // z comes from the kernel before this one
    const uint32_t b_bytes = static_cast<uint32_t>(kTileM * p.R_pad * 2), z_bytes = static_cast<uint32_t>(p.R_pad) * 4;
    uint32_t stage = 0, phase = 0, info = 0;  // lane l: rank, tokens and first position of the stage l of the next 32
    int32_t adapter = 0;                      // and its adapter
    int live = 0;
    const int n_blocks = sh.groups.n_blocks;
    for (int s = 0; ok && s < n_blocks; ++s) {
      if ((s & 31) == 0 && s + lane < n_blocks) {
        info = stage_info(sh, s + lane);
        adapter = sh.groups.adapter[sh.groups.block_group[s + lane]];
      }
      const uint32_t mine = __shfl_sync(0xffffffffu, info, s & 31);
      const int32_t a = __shfl_sync(0xffffffffu, adapter, s & 31);
      const int rank = mine & 255, nt = (mine >> 8) & 255, pos = mine >> 16;
      if (rank == 0) continue;  // an empty slot: its tokens stay base-only
      if ((live++ & 1) == half) {
        if (ptx::elect_one()) {
          ok = ptx::mbar_wait(&sh.bempty[stage], phase ^ 1, wl) && !sh.abort_flag;
          if (ok) {
            uint8_t *dst = exp_ring + static_cast<size_t>(stage) * p.exp_bytes;
            ptx::mbar_arrive_expect_tx(&sh.bfull[stage], b_bytes + nt * z_bytes);
            ptx::tma_load_3d(dst, &p.b, &sh.bfull[stage], 0, row0, a);
            for (int q = 0; q < nt; ++q)
              ptx::bulk_load_1d(dst + b_bytes + q * z_bytes, p.z + static_cast<size_t>(t0 + sh.groups.tok[pos + q]) * p.R_pad,
                                z_bytes, &sh.bfull[stage]);
          }
        }
        ok = __all_sync(0xffffffffu, ok);
      }
      if (++stage == nexp) {
        stage = 0;
        phase ^= 1;
      }
    }
  } else if (warp >= 4) {
    // ------------------------------------------------------------ u-batches and expand (warps 4..11)
    const int quad = warp & 3, row_in_tile = quad * 32 + lane, half = (warp - 4) >> 2, etid = tid - 128;
    const uint32_t texp = tmem_exp + (static_cast<uint32_t>(quad * 32) << 16);
    derive_groups<kExpTok, 1, kExpandThreads>(sh.groups, p.ids + t0, n_own, p.n_slots, etid);
    if (etid < sh.groups.n_groups) {
      const int32_t a = sh.groups.adapter[etid];
      sh.rank[etid] = EL_CHECK(p.status, a >= 0 && a < p.n_slots, 1) ? static_cast<uint8_t>(p.slots[a].rank) : 0;
    }
    __syncwarp();
    for (int32_t c = half * 32; c < n_own; c += 64) ptx::tmem_fill_32x32(texp + c, 0.f);
    ptx::tmem_st_wait();
    ptx::tc_fence_before_sync();
    ptx::named_barrier<1, kExpandThreads>();
    ptx::tc_fence_after_sync();
    if (etid == 0) ptx::mbar_arrive(&sh.groups_ready);
    const uint32_t b_bytes = static_cast<uint32_t>(kTileM * p.R_pad * 2);
    const int sw = row_swizzle(row_in_tile, p.R_pad);
    uint32_t stage = 0, phase = 0, info = 0;  // lane l: rank, tokens and first position of the stage l of the next 32
    int live = 0;
    const int n_blocks = sh.groups.n_blocks;
    for (int s = 0; s < n_blocks; ++s) {
      if ((s & 31) == 0 && s + lane < n_blocks) info = stage_info(sh, s + lane);
      const uint32_t mine = __shfl_sync(0xffffffffu, info, s & 31);
      const int rank = mine & 255, nt = (mine >> 8) & 255, pos = mine >> 16;
      if (rank == 0) continue;
      if ((live++ & 1) == half) {  // the groups of four warps take every other stage
        // (the first one is for z, too: it ends behind the shrink)
        const bool there = live <= 2 ? ptx::mbar_wait_timed(&sh.bfull[stage], phase, wl) : ptx::mbar_wait(&sh.bfull[stage], phase, wl);
        if (!__all_sync(0xffffffffu, there && !sh.abort_flag)) {
          ok = false;
          break;
        }
        const uint8_t *src = exp_ring + static_cast<size_t>(stage) * p.exp_bytes;
        const uint8_t *brow = src + row_in_tile * p.R_pad * 2;
        const uint32_t z = ptx::smem_u32(src + b_bytes);
        const uint32_t z_bytes = static_cast<uint32_t>(p.R_pad) * 4;
        if (rank <= 8) expand_stage<1>(brow, sw, z, z_bytes, rank, nt, texp, sh.groups.tok + pos);
        else if (rank <= 16) expand_stage<2>(brow, sw, z, z_bytes, rank, nt, texp, sh.groups.tok + pos);
        else if (rank <= 32) expand_stage<4>(brow, sw, z, z_bytes, rank, nt, texp, sh.groups.tok + pos);
        else expand_stage<8>(brow, sw, z, z_bytes, rank, nt, texp, sh.groups.tok + pos);
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&sh.bempty[stage]);
      }
      if (++stage == nexp) {
        stage = 0;
        phase ^= 1;
      }
    }
    __syncwarp();
    ptx::tmem_st_wait();
    if (!__all_sync(0xffffffffu, ptx::mbar_wait(&sh.tfull, 0, wl))) ok = false;
  }
  if (!ok) {
    sh.abort_flag = 1;
    atomicOr(p.status, EDGELORA_STATUS_TIMEOUT);
    ptx::settle();
  }
  __syncwarp();
  ptx::tc_fence_before_sync();
  __syncthreads();  // the accumulator and the expand are complete, the rings idle
  ptx::tc_fence_after_sync();

  // ---------------------------------------------------------------- exchange of the parts, y
  // Each part's sums of the other owners' columns, as [owner][quad][row][4 tokens] in the memory of the rings, go to the owners
  // in one bulk copy each as soon as every CTA of the cluster is there.  (Stores of the threads into the other CTAs' memory took
  // 6 us for 256 columns.)
  const uint32_t slot_bytes = static_cast<uint32_t>(per) * (kTileM * 16);
  uint8_t *to_send = smem, *received = smem + static_cast<size_t>(p.parts - 1) * slot_bytes;
  const int quad = warp & 3, row_in_tile = quad * 32 + lane, half = (warp - 4) >> 2;
  const uint32_t lanes = static_cast<uint32_t>(quad * 32) << 16;
  const bool base = kb1 > kb0;
  auto load16 = [&](uint32_t from, float (&v)[16]) {
    ptx::tmem_ld_32x16(from + lanes, v);
    ptx::tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 16; ++j) ptx::tmem_loaded(v[j]);
  };
  if (p.parts > 1) {
    if (warp >= 4) {
      for (int32_t q = half * 4; q < n_quads; q += 8) {  // the warps of a lane quadrant take every other 16 columns
        if (q >= q0 && q + 4 <= q0 + nq) continue;
        float v[16];
        load16(tmem_acc + q * 4, v);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int32_t owner = (q + j) / per, at = q + j - owner * per;
          if (q + j < n_quads && owner != part)
            *reinterpret_cast<float4 *>(to_send + (owner - (owner > part ? 1 : 0)) * slot_bytes + (at * kTileM + row_in_tile) * 16) =
                base ? make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
      ptx::fence_proxy_async();
      ptx::tc_fence_before_sync();
    }
    __syncwarp();
    ptx::cluster_sync_all();
    ptx::tc_fence_after_sync();
    if (tid == 0) {
      ptx::mbar_arrive_expect_tx(&sh.parts, static_cast<uint32_t>((p.parts - 1) * nq * (kTileM * 16)));
      for (int32_t o = 0; o < p.parts; ++o) {
        const int32_t n = min(per, n_quads - o * per);
        if (o == part || n <= 0) continue;
        ptx::bulk_copy_cluster(ptx::map_to_rank(ptx::smem_u32(received + (part - (part > o ? 1 : 0)) * slot_bytes), o),
                               to_send + (o - (o > part ? 1 : 0)) * slot_bytes, static_cast<uint32_t>(n * (kTileM * 16)),
                               ptx::map_to_rank(ptx::smem_u32(&sh.parts), o));
      }
    }
    __syncwarp();
  }
  if (warp >= 4) {
    ptx::pdl_wait_prior_grids();  // earlier kernels may still read y
    if (p.parts > 1 && !__all_sync(0xffffffffu, ptx::mbar_wait(&sh.parts, 0, max(wl, ptx::kSettleCycles))))
      atomicOr(p.status, EDGELORA_STATUS_TIMEOUT);
    const int32_t row = row0 + row_in_tile;
    __syncwarp();
    for (int32_t q = half * 4; q < nq; q += 8) {
      float own[16], e[16], v[16];
      ptx::tmem_ld_32x16(tmem_exp + lanes + q * 4, e);
      load16(tmem_acc + (q0 + q) * 4, own);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        ptx::tmem_loaded(e[j]);
        if (!base) own[j] = 0.f;
        v[j] = part == 0 ? own[j] : 0.f;
      }
      for (int32_t c = 0; c < p.parts; ++c) {  // the parts in order
        if (c == part) {
          if (c > 0) {
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] += own[j];
          }
          continue;
        }
        const uint8_t *from = received + (c - (c > part ? 1 : 0)) * slot_bytes + (q * kTileM + row_in_tile) * 16;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (q + j < nq) {
            const float4 w = *reinterpret_cast<const float4 *>(from + j * (kTileM * 16));
            v[4 * j] += w.x; v[4 * j + 1] += w.y; v[4 * j + 2] += w.z; v[4 * j + 3] += w.w;
          }
        }
      }
      if (row < p.h_out) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (q * 4 + j < n_own)
            p.y[static_cast<size_t>(t0 + q * 4 + j) * p.h_out + row] =
                static_cast<uint16_t>(ptx::pack_bf16x2(v[j] + e[j], 0.f) & 0xFFFFu);
      }
      __syncwarp();
    }
    ptx::tc_fence_before_sync();
  }
  __syncwarp();
  if (p.parts > 1)
    ptx::cluster_sync_all();  // what this CTA sent has arrived
  else
    __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tmem_acc, static_cast<uint32_t>(p.tmem_cols));
  }
}

DecTileShape decode_tile_shape(int32_t N, int32_t R_pad) {
  DecTileShape s{};
  const size_t stage = kWBytes + static_cast<size_t>(N) * kBlockK * 2;
  s.exp_bytes = (kTileM * R_pad * 2 + kExpTok * R_pad * 4 + 1023) & ~1023;
  s.stages = std::min<int32_t>(kTileMaxStages, static_cast<int32_t>((kRingBytes - static_cast<size_t>(kExpStages) * s.exp_bytes) / stage));
  s.tmem_cols = 32;
  while (s.tmem_cols < 2 * ((N + 31) & ~31)) s.tmem_cols <<= 1;
  return s;
}

bool decode_tile_parts_fit(int32_t T, int32_t parts) {
  const size_t quads = (T + 3) / 4, per = (quads + parts - 1) / parts;
  return 2 * (parts - 1) * per * kTileM * 16 <= kRingBytes;
}

cudaError_t decode_tile_set_smem_limit() {
  return cudaFuncSetAttribute(decode_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kTileSmemBudget));
}

cudaError_t launch_decode_tile(const DecTile &p, bool pdl, cudaStream_t stream) {
  const int32_t tiles = (p.h_out + kTileM - 1) / kTileM;
  return launch_ex(decode_tile_kernel, dim3(tiles * p.parts), dim3(kThreads), kTileSmemBudget, stream, pdl, p.parts, p);
}

int32_t decode_tile_max_clusters(int32_t parts) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(parts) * 64);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kTileSmemBudget;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(parts);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, decode_tile_kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

}  // namespace edgelora
