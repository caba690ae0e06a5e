// Decode-sized batches (at most 256 tokens) through a run of linear sites that see the same batch (paper Section 3.4: the
// base product W [x_0 .. x_n] batched over every token, plus s_a B_a A_a x per token, y written once), in two launches for
// the whole run: the shrink of every site, then every site's base product with the expand.
//
// Base product: D[128 x N] (fp32, in tensor memory) = R[128 x K] * C[N x K]^T, R = 128 rows of W, C = all tokens, K blocks
// of 64 from a TMA ring.  What bounds it is the stream of W.  The K blocks of all tiles of all sites, and the expand's share
// of each tile, form one list of units that is cut into equal runs, one per CTA of a persistent grid: no SM idles in the
// last wave of a site, and ramp-up and drain are paid once per launch.  A run cuts a tile at its two ends only; the parts of
// such a tile go to fp32 planes in global memory, and the CTA that arrives last adds them in the order of the runs (nobody
// waits for another CTA).
//
// Expand: on the CUDA cores from fp32 z, row by row for the tokens of an adapter, beside the stream of W: the B_a rows of
// the tile and the z rows of up to eight tokens of the adapter come through a ring of their own, the dot products wait in
// tensor memory until the accumulator is complete.  An adapter's values reach the rows of its own tokens only.
//
// 28 sites of four decoder layers (4096, 1024, 14336 wide), 27 tokens on 18 adapters of rank 8 to 32: 337 us for 1.93 GB
// that cannot be done without (2.04 GB as the B blocks are padded: 6.1 TB/s), 416 us with two launches per site; seven
// sites of a layer 1024 wide, one token: 21 us, 45 before.  64 tokens: 400 us, 565 before; 256 tokens through two layers:
// 483 us, 671 before.
//
// Warp roles of the base kernel: warp 0 issues the TMA loads of W and x, warp 1 owns tensor memory and issues the MMAs,
// warp 2 issues the copies of the expand, warps 4..7 (the four lane quadrants) work out the expand and write y.  Every
// mbarrier wait is bounded; on a timeout every site's status word gets EDGELORA_STATUS_TIMEOUT and all roles leave.
#include <algorithm>

#include "decode_route.cuh"
#include "decode_sites.h"
#include "expand.cuh"
#include "launch.cuh"
#include "ptx.cuh"
#include "shrink_rows.cuh"
#include "units.h"

namespace edgelora {

namespace {

constexpr uint32_t kWBytes = kTileM * kBlockK * 2;

struct DecShared {
  uint64_t full[kDecMaxStages];          // TMA -> MMA
  uint64_t empty[kDecMaxStages];         // MMA -> TMA
  uint64_t bfull[kDecMaxExpStages];      // copies of the expand -> epilogue
  uint64_t bempty[kDecMaxExpStages];     // epilogue -> copies of the expand
  uint64_t tfull[2], tempty[2];          // MMA -> epilogue, epilogue -> MMA
  uint64_t lfull[2], lempty[2];          // ranks of a site: epilogue -> warp 2, warp 2 -> epilogue
  uint32_t tmem_slot;
  volatile uint32_t abort_flag;
  int32_t site_end[kDecSites];           // units of the sites up to each
  uint8_t rank[2][kDecodeMaxT];          // rank of every group's adapter at the site of a piece
  Groups groups;
};
static_assert(sizeof(DecShared) <= kDecTailBytes, "tail of the shared memory");

// A barrier of the epilogue warps; every thread learns whether any of them passed true.
__device__ __forceinline__ bool epilogue_any(bool v) {
  uint32_t r;
  __syncwarp();
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, 1, 128, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(v ? 1u : 0u)
      : "memory");
  return r != 0;
}

// Stages of the units [e0, e1).
__device__ __forceinline__ int32_t first_stage(int32_t unit, int32_t n_stages, int32_t R_pad) {
  return min(unit * (64 >> (31 - __clz(R_pad))), n_stages);
}

// The stage's tokens, four, two or one at a time, into the columns from `taddr` on.
template <int kChunks>
__device__ __forceinline__ void expand_stage(const uint8_t *brow, int sw, uint32_t z, uint32_t z_bytes, int rank, int nt,
                                             uint32_t taddr) {
  float acc[4];
#pragma unroll 1
  for (; nt >= 4; nt -= 4, z += 4 * z_bytes, taddr += 4) {
    expand_dots<kChunks, 4>(brow, sw, z, z_bytes, rank, acc);
    ptx::tmem_st_32x4(taddr, acc);
  }
  if (nt & 2) {
    expand_dots<kChunks, 2>(brow, sw, z, z_bytes, rank, acc);
    ptx::tmem_st_32x2(taddr, acc);
    z += 2 * z_bytes;
    taddr += 2;
  }
  if (nt & 1) {
    expand_dots<kChunks, 1>(brow, sw, z, z_bytes, rank, acc);
    ptx::tmem_st_32x1(taddr, acc);
  }
}
// Tensor-memory column of the expand of token t, or -1 when the piece at hand has none for it: positions [p0, p1) of the
// tokens in the order of their adapters, on slots that are loaded.
__device__ __forceinline__ int expand_column(const Groups &g, const uint8_t *rank, int t, int T, int p0, int p1) {
  if (t >= T || g.id[t] < 0) return -1;
  const int p = g.pos[t];
  return p >= p0 && p < p1 && rank[g.group[t]] > 0 ? p : -1;
}
// The expand's values of kN tokens, token j's column held by lane j, added to v.
template <int kN>
__device__ __forceinline__ void add_expand(uint32_t texp, int column, float *v) {
  if (__ballot_sync(0xffffffffu, column >= 0) == 0) return;
  float e[kN];
#pragma unroll
  for (int j = 0; j < kN; ++j) {
    const int c = __shfl_sync(0xffffffffu, column, j);
    e[j] = 0.f;
    if (c >= 0) ptx::tmem_ld_32x1(texp + c, e[j]);
  }
  ptx::tmem_ld_wait();
#pragma unroll
  for (int j = 0; j < kN; ++j) {
    ptx::tmem_loaded(e[j]);
    v[j] += e[j];
  }
}

}  // namespace

__global__ void __launch_bounds__(kDecThreads, 1) decode_sites_kernel(const __grid_constant__ DecBatch b) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t x_bytes = static_cast<uint32_t>(b.N) * (kBlockK * 2), stage_bytes = kWBytes + x_bytes;
  const uint32_t nstages = static_cast<uint32_t>(b.stages), nexp = static_cast<uint32_t>(b.exp_stages);
  uint8_t *exp_ring = smem + static_cast<size_t>(nstages) * stage_bytes;
  DecShared &sh = *reinterpret_cast<DecShared *>(exp_ring + static_cast<size_t>(nexp) * b.exp_bytes);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long wl = b.wait_cycles;
  const int32_t Nc = (b.N + 31) & ~31;  // tensor memory columns of an accumulator
  const int32_t me = static_cast<int32_t>(blockIdx.x);

  if (tid == 0) {
    ptx::prefetch_tensormap(&b.x[b.site[0].x_index]);
    for (uint32_t s = 0; s < nstages; ++s) {
      ptx::mbar_init(&sh.full[s], 1);
      ptx::mbar_init(&sh.empty[s], 1);
    }
    for (uint32_t s = 0; s < nexp; ++s) {
      ptx::mbar_init(&sh.bfull[s], 1);
      ptx::mbar_init(&sh.bempty[s], 4);  // one arrival per epilogue warp
    }
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&sh.tfull[i], 1);
      ptx::mbar_init(&sh.tempty[i], 4);
      ptx::mbar_init(&sh.lfull[i], 1);
      ptx::mbar_init(&sh.lempty[i], 1);
    }
    sh.abort_flag = 0;
    ptx::fence_barrier_init();
  }
  if (warp == 1) {
    ptx::tmem_alloc(&sh.tmem_slot, static_cast<uint32_t>(b.tmem_cols));
    ptx::tmem_relinquish();
  }
  if (warp >= 4) derive_groups<kExpTok, 1, 128>(sh.groups, b.ids, b.T, b.n_slots, tid - 128);
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  ptx::pdl_launch_dependents();
  const int32_t n_stages = sh.groups.n_blocks, n_groups = sh.groups.n_groups;
  if (warp == 0) {  // units of the sites up to each
    int32_t u = 0;
    if (lane < b.n_sites) {
      const DecSite &st = b.site[lane];
      u = (st.h_out + kTileM - 1) / kTileM * (st.kb + expand_units(n_stages, st.R_pad));
    }
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int32_t o = __shfl_up_sync(0xffffffffu, u, d);
      if (lane >= d) u += o;
    }
    if (lane < b.n_sites) sh.site_end[lane] = u;
  }
  __syncthreads();
  const uint32_t tmem_base = sh.tmem_slot, tmem_exp = tmem_base + static_cast<uint32_t>(b.n_acc * Nc);
  const int32_t n_units = sh.site_end[b.n_sites - 1];
  const int32_t n_runs = run_count(n_units, static_cast<int32_t>(gridDim.x));
  const Runs runs(n_units, n_runs);
  const int32_t u_begin = me < n_runs ? runs.begin(me) : n_units, u_end = me < n_runs ? runs.begin(me + 1) : n_units;
  int32_t site = 0;
  bool ok = true;
  // Roles walk the pieces of the run: for (u = u_begin; u < u_end; u += units done).
  auto next_piece = [&](int32_t &u) {
    const Piece p = piece_at(
        u, u_end, sh.site_end, [&](int32_t s) { return expand_units(n_stages, b.site[s].R_pad); },
        [&](int32_t s) { return b.site[s].kb; }, site);
    u += p.size();
    return p;
  };

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (W and x)
    if (ptx::elect_one()) {
      uint32_t stage = 0, phase = 0;
      for (int32_t u = u_begin; ok && u < u_end;) {
        const Piece p = next_piece(u);
        const DecSite &st = b.site[p.s];
        for (int32_t kb = p.kb0; kb < p.kb1; ++kb) {
          if (!ptx::mbar_wait(&sh.empty[stage], phase ^ 1, wl) || sh.abort_flag) {
            ok = false;
            break;
          }
          uint8_t *sr = smem + static_cast<size_t>(stage) * stage_bytes;
          ptx::mbar_arrive_expect_tx(&sh.full[stage], stage_bytes);
          ptx::tma_load_2d(sr, &st.w, &sh.full[stage], kb * kBlockK, p.tile * kTileM);
          ptx::tma_load_2d(sr + kWBytes, &b.x[st.x_index], &sh.full[stage], kb * kBlockK, 0);
          if (++stage == nstages) {
            stage = 0;
            phase ^= 1;
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (ptx::elect_one()) {
      const uint32_t idesc = ptx::umma_idesc_bf16(kTileM, static_cast<uint32_t>(b.N));
      uint32_t stage = 0, phase = 0, it = 0;
      for (int32_t u = u_begin; ok && u < u_end;) {
        const Piece p = next_piece(u);
        if (p.kb1 == p.kb0) continue;
        const uint32_t acc = b.n_acc == 2 ? it & 1 : 0, par = b.n_acc == 2 ? (it >> 1) & 1 : it & 1;
        ++it;
        if (!ptx::mbar_wait(&sh.tempty[acc], par ^ 1, wl) || sh.abort_flag) {
          ok = false;
          break;
        }
        ptx::tc_fence_after_sync();
        const uint32_t tmem_d = tmem_base + acc * static_cast<uint32_t>(Nc);
        for (int32_t kb = p.kb0; kb < p.kb1; ++kb) {
          if (!ptx::mbar_wait(&sh.full[stage], phase, wl) || sh.abort_flag) {
            ok = false;
            break;
          }
          ptx::tc_fence_after_sync();
          const uint32_t sr = ptx::smem_u32(smem + static_cast<size_t>(stage) * stage_bytes);
          const uint64_t da = ptx::umma_desc_k128(sr), db = ptx::umma_desc_k128(sr + kWBytes);
#pragma unroll
          for (int k = 0; k < kBlockK / kUmmaK; ++k)
            ptx::umma_bf16(tmem_d, da + 2 * k, db + 2 * k, idesc, (kb > p.kb0 || k > 0) ? 1u : 0u);
          ptx::umma_commit(&sh.empty[stage]);
          if (++stage == nstages) {
            stage = 0;
            phase ^= 1;
          }
        }
        if (ok) ptx::umma_commit(&sh.tfull[acc]);
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------ copies of the expand (B_a rows and z)
    if (ptx::elect_one()) {
      uint32_t stage = 0, phase = 0, it = 0;
      bool waited = false;
      for (int32_t u = u_begin; ok && u < u_end;) {
        const Piece p = next_piece(u);
        if (p.e1 == p.e0) continue;
        const DecSite &st = b.site[p.s];
        const uint32_t buf = it & 1;
        if (!ptx::mbar_wait(&sh.lfull[buf], (it >> 1) & 1, wl)) {
          ok = false;
          break;
        }
        ++it;
        if (!waited) {  // z comes from the kernel before this one
          ptx::pdl_wait_prior_grids();
          waited = true;
        }
        const uint32_t b_bytes = static_cast<uint32_t>(kTileM * st.R_pad * 2), z_bytes = static_cast<uint32_t>(st.R_pad) * 4;
        const int32_t s1 = first_stage(p.e1, n_stages, st.R_pad);
        for (int32_t s = first_stage(p.e0, n_stages, st.R_pad); s < s1; ++s) {
          const int g = sh.groups.block_group[s], pos = sh.groups.block_pos[s];
          if (sh.rank[buf][g] == 0) continue;  // an empty slot: its tokens stay base-only
          const int32_t a = sh.groups.adapter[g];
          const int nt = min(kExpTok, sh.groups.start[g + 1] - pos);
          if (!ptx::mbar_wait(&sh.bempty[stage], phase ^ 1, wl) || sh.abort_flag) {
            ok = false;
            break;
          }
          uint8_t *dst = exp_ring + static_cast<size_t>(stage) * b.exp_bytes;
          ptx::mbar_arrive_expect_tx(&sh.bfull[stage], b_bytes + nt * z_bytes);
          ptx::tma_load_3d(dst, &st.b, &sh.bfull[stage], 0, p.tile * kTileM, a);
          for (int q = 0; q < nt; ++q)
            ptx::bulk_load_1d(dst + b_bytes + q * z_bytes, st.z + static_cast<size_t>(sh.groups.tok[pos + q]) * st.R_pad, z_bytes,
                              &sh.bfull[stage]);
          if (++stage == nexp) {
            stage = 0;
            phase ^= 1;
          }
        }
        ptx::mbar_arrive(&sh.lempty[buf]);
      }
    }
  } else if (warp >= 4) {
    // ------------------------------------------------------------ expand and epilogue (warps 4..7)
    const int quad = warp & 3, row_in_tile = quad * 32 + lane, etid = tid - 128;
    const uint32_t lanes = static_cast<uint32_t>(quad * 32) << 16;
    uint32_t stage = 0, phase = 0, it = 0, lit = 0;
    bool waited = false;
    for (int32_t u = u_begin; u < u_end;) {
      const Piece p = next_piece(u);
      const DecSite &st = b.site[p.s];
      const int32_t row = p.tile * kTileM + row_in_tile;
      const bool expand = p.e1 > p.e0, base = p.kb1 > p.kb0;
      const uint32_t buf = lit & 1;
      if (expand) {
        ok = __all_sync(0xffffffffu, ok && ptx::mbar_wait(&sh.lempty[buf], ((lit >> 1) & 1) ^ 1, wl) && !sh.abort_flag);
        ++lit;
        for (int g = etid; ok && g < n_groups; g += 128) {
          const int32_t a = sh.groups.adapter[g];
          sh.rank[buf][g] = EL_CHECK(st.status, a >= 0 && a < b.n_slots, 1) ? static_cast<uint8_t>(st.slots[a].rank) : 0;
        }
      }
      if (epilogue_any(!ok)) {  // (the four warps leave together: none waits here for one that gave up)
        ok = false;
        break;
      }
      int p0 = 0, p1 = 0;  // positions of the piece's tokens
      if (expand) {
        if (etid == 0) ptx::mbar_arrive(&sh.lfull[buf]);
        const uint32_t b_bytes = static_cast<uint32_t>(kTileM * st.R_pad * 2);
        const int sw = row_swizzle(row_in_tile, st.R_pad);
        const int32_t s0 = first_stage(p.e0, n_stages, st.R_pad), s1 = first_stage(p.e1, n_stages, st.R_pad);
        p0 = s0 < n_stages ? sh.groups.block_pos[s0] : b.T;
        p1 = s1 < n_stages ? sh.groups.block_pos[s1] : b.T;
        uint32_t info = 0;  // lane l: rank, tokens and first position of the stage l of the next 32
        for (int32_t s = s0; s < s1; ++s) {
          const int l = (s - s0) & 31;
          if (l == 0 && s + lane < s1) {
            const int g = sh.groups.block_group[s + lane], pos = sh.groups.block_pos[s + lane];
            info = sh.rank[buf][g] | min(kExpTok, sh.groups.start[g + 1] - pos) << 8 | pos << 16;
          }
          const uint32_t mine = __shfl_sync(0xffffffffu, info, l);
          const int rank = mine & 255, nt = (mine >> 8) & 255, pos = mine >> 16;
          if (rank == 0) continue;
          if (!__all_sync(0xffffffffu, ptx::mbar_wait(&sh.bfull[stage], phase, wl) && !sh.abort_flag)) {
            ok = false;
            break;
          }
          const uint8_t *src = exp_ring + static_cast<size_t>(stage) * b.exp_bytes;
          const uint8_t *brow = src + row_in_tile * st.R_pad * 2;
          const uint32_t z = ptx::smem_u32(src + b_bytes), taddr = tmem_exp + lanes + pos;
          const uint32_t z_bytes = static_cast<uint32_t>(st.R_pad) * 4;
          if (rank <= 8) expand_stage<1>(brow, sw, z, z_bytes, rank, nt, taddr);
          else if (rank <= 16) expand_stage<2>(brow, sw, z, z_bytes, rank, nt, taddr);
          else if (rank <= 32) expand_stage<4>(brow, sw, z, z_bytes, rank, nt, taddr);
          else expand_stage<8>(brow, sw, z, z_bytes, rank, nt, taddr);
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&sh.bempty[stage]);
          __syncwarp();
          if (++stage == nexp) {
            stage = 0;
            phase ^= 1;
          }
        }
        ptx::tmem_st_wait();
      }
      uint32_t acc_i = 0;
      if (ok && base) {
        acc_i = b.n_acc == 2 ? it & 1 : 0;
        const uint32_t par = b.n_acc == 2 ? (it >> 1) & 1 : it & 1;
        ++it;
        ok = __all_sync(0xffffffffu, ptx::mbar_wait(&sh.tfull[acc_i], par, wl) && !sh.abort_flag);
        ptx::tc_fence_after_sync();
      }
      if (!ok) {
        sh.abort_flag = 1;
        continue;
      }
      if (!waited) {  // earlier kernels may still read y and the planes
        ptx::pdl_wait_prior_grids();
        waited = true;
      }
      const int32_t c0 = runs.of(p.first), c1 = runs.of(p.first + p.units - 1);  // the runs that share the tile
      const size_t plane = static_cast<size_t>(b.N) * kTileM;
      float *mine = b.partial + (2 * static_cast<size_t>(me) + (me == c0 ? 1 : 0)) * plane + row_in_tile;
      const uint32_t tacc = tmem_base + lanes + acc_i * static_cast<uint32_t>(Nc), texp = tmem_exp + lanes;
      for (int32_t n0 = 0; n0 < b.N; n0 += 32) {
        float v[32];
        __syncwarp();
        if (base) {
          ptx::tmem_ld_32x32(tacc + n0, v);
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = 0.f;
        }
        if (expand) add_expand<32>(texp, expand_column(sh.groups, sh.rank[buf], n0 + lane, b.T, p0, p1), v);
        if (base && n0 + 32 >= b.N) {  // the accumulator is read
          ptx::tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&sh.tempty[acc_i]);
        }
        if (c0 == c1) {
          if (row < st.h_out) {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (n0 + j < b.T)
                st.y[static_cast<size_t>(n0 + j) * st.h_out + row] =
                    static_cast<uint16_t>(ptx::pack_bf16x2(v[j], 0.f) & 0xFFFFu);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (n0 + j < b.T) mine[(n0 + j) * kTileM] = v[j];
        }
      }
      if (c0 != c1) {
        // The warp that arrives last for these 32 rows of the tile adds the planes in the order of the runs.
        __threadfence();
        __syncwarp();
        int32_t old = 0;
        if (lane == 0) old = atomicAdd(&b.arrivals[c0 * 4 + quad], 1);
        old = __shfl_sync(0xffffffffu, old, 0);
        if (old == c1 - c0) {
          __threadfence();
          for (int32_t t0 = 0; t0 < b.T; t0 += 16) {
            float v[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = 0.f;
#pragma unroll 2
            for (int32_t c = c0; c <= c1; ++c) {
              const float *from = b.partial + (2 * static_cast<size_t>(c) + (c == c0 ? 1 : 0)) * plane + row_in_tile;
#pragma unroll
              for (int j = 0; j < 16; ++j) v[j] += t0 + j < b.T ? __ldcg(from + (t0 + j) * kTileM) : 0.f;
            }
            if (row < st.h_out) {
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (t0 + j < b.T)
                  st.y[static_cast<size_t>(t0 + j) * st.h_out + row] =
                      static_cast<uint16_t>(ptx::pack_bf16x2(v[j], 0.f) & 0xFFFFu);
            }
          }
        }
      }
    }
  }
  if (!ok) {  // what this CTA leaves undone may belong to any site
    sh.abort_flag = 1;
    for (int32_t s = 0; s < b.n_sites; ++s) atomicOr(b.site[s].status, EDGELORA_STATUS_TIMEOUT);
    ptx::settle();
  }
  __syncwarp();
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tmem_base, static_cast<uint32_t>(b.tmem_cols));
  }
}

// ------------------------------------------------------------------------------------------------------- shrink
//
// z[t] = s_a A_a x[t] for the tokens of every site, on the CUDA cores (see shrink.cu for the arithmetic and the rings).
// Work items (site, block of up to four tokens of an adapter, eight rank rows, K chunk) belong to single warps; a CTA's
// items are dealt to it round-robin and drawn by its warps from a counter in shared memory.  The last CTA publishes the
// plan.
constexpr int kDecShrinkDepth = 2;
constexpr size_t kDecShrinkRing = static_cast<size_t>(kDecThreads / 32) * kDecShrinkDepth * kDsStageBytes;

__global__ void __launch_bounds__(kDecThreads, 2) decode_sites_shrink_kernel(const __grid_constant__ DecShrinkBatch b) {
  extern __shared__ __align__(128) uint8_t s_dyn[];  // rings, then a byte per (site, group): the rank
  __shared__ uint64_t s_bars[kDecThreads / 32][kDsMaxDepth];
  __shared__ __align__(16) Groups s_groups;
  __shared__ int32_t s_end[kDecSites];
  __shared__ int32_t s_ticket;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  ptx::pdl_launch_dependents();
  if (tid == 0) s_ticket = 0;
  if (lane < kDsMaxDepth) {  // every warp sets up its own ring barriers
    ptx::mbar_init(&s_bars[warp][lane], 1);
    ptx::fence_barrier_init();
  }
  const bool bad = derive_groups<kDsTok, 1, kDecThreads>(s_groups, b.ids, b.T, b.n_slots, tid);
  const int any_bad = __syncthreads_or(bad ? 1 : 0), G = s_groups.n_groups, NB = s_groups.n_blocks;
  uint8_t *s_rank = s_dyn + kDecShrinkRing;  // [site][G]
  if (blockIdx.x == gridDim.x - 1) {
    // the plan in canonical order, and the arrival counters of the launch behind this one
    publish_decode_plan(b.pv, s_groups.id[tid], b.T, any_bad, 1, s_groups.id, s_groups.cnt, s_groups.wt);  // waits for the kernels before
    for (int i = tid; i < b.n_zero; i += kDecThreads) b.zero[i] = 0;
    return;
  }
  for (int i = tid; i < b.n_sites * G; i += kDecThreads) {
    const int s = i / G;
    s_rank[i] = static_cast<uint8_t>(b.site[s].slots[s_groups.adapter[i - s * G]].rank);
  }
  if (warp == 0) {
    int32_t n = lane < b.n_sites ? NB * (b.site[lane].R_pad >> 3) * b.site[lane].ks : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int32_t o = __shfl_up_sync(0xffffffffu, n, d);
      if (lane >= d) n += o;
    }
    if (lane < b.n_sites) s_end[lane] = n;
  }
  __syncthreads();
  const int n_items = s_end[b.n_sites - 1], workers = static_cast<int>(gridDim.x) - 1;
  uint8_t *ring = s_dyn + static_cast<size_t>(warp) * kDecShrinkDepth * kDsStageBytes;
  uint64_t *bars = s_bars[warp];
  uint32_t phase = 0;
  bool ok = true, waited = false;
  int site = 0;
  while (ok) {
    int item = 0;
    if (lane == 0) item = static_cast<int>(blockIdx.x) + atomicAdd(&s_ticket, 1) * workers;
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= n_items) break;
    while (item >= s_end[site]) ++site;
    const DecShrinkSite &st = b.site[site];
    const int local = item - (site > 0 ? s_end[site - 1] : 0);
    // (chunk c takes the K steps c, c + ks, ..: see decode_shrink_kernel)
    const int c = local % st.ks, br = local / st.ks, n_rgn = st.R_pad >> 3;
    const int bi = br / n_rgn, rg = br - bi * n_rgn;
    const int gi = s_groups.block_group[bi], t0 = s_groups.block_pos[bi];
    const int g_begin = s_groups.start[gi], g_end = s_groups.start[gi + 1];
    const int ad = s_groups.adapter[gi], rank = s_rank[site * G + gi];
    if (rank == 0 && lane == 0 && c == 0 && rg == 0 && t0 == g_begin) atomicOr(st.status, EDGELORA_STATUS_SLOT_EMPTY);
    if (rg * 8 >= rank) continue;  // zero padding of the block
    const float scale = st.slots[ad].scale;
    const int nt = min(kDsTok, g_end - t0);
    float acc[8 * kDsTok];
#pragma unroll
    for (int i = 0; i < 8 * kDsTok; ++i) acc[i] = 0.f;
    int32_t tok[kDsTok];
#pragma unroll
    for (int q = 0; q < kDsTok; ++q) tok[q] = s_groups.tok[t0 + min(q, nt - 1)];
    const CUtensorMap *mx = &b.x[st.x_index];
#define EDGELORA_ROWS(NT)                                                                                            \
  shrink_rows8<NT, kDecShrinkDepth, false>(&st.a, &st.a, mx, ad, rg * 8, tok, c, st.n_ksteps, st.ks, ring, bars, phase, \
                                           lane, acc)
    if (nt == 1) ok = EDGELORA_ROWS(1);
    else if (nt == 2) ok = EDGELORA_ROWS(2);
    else if (nt == 3) ok = EDGELORA_ROWS(3);
    else ok = EDGELORA_ROWS(4);
#undef EDGELORA_ROWS
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) break;
    sum_over_lanes(acc, lane);  // value L: row L / 4, token L % 4
    if (!waited) {  // first write of this warp to memory that earlier kernels may read
      ptx::pdl_wait_prior_grids();
      waited = true;
    }
    const size_t zplane = static_cast<size_t>(st.max_tokens) * st.R_pad;
    const int q = lane & 3, r = rg * 8 + (lane >> 2);
    if (q < nt && EL_CHECK(st.status, s_groups.tok[t0 + q] < st.max_tokens && ad >= 0 && ad < b.n_slots, 20))
      st.zws[(st.ks > 1 ? c : kMaxZSplits) * zplane + static_cast<size_t>(s_groups.tok[t0 + q]) * st.R_pad + r] =
          scale * acc[0];
    if (st.ks > 1) {  // the warp that completes a (group, eight rows) adds the K chunks in order
      const int arrivals = st.ks * ((g_end - g_begin + kDsTok - 1) / kDsTok);
      __syncwarp();  // the lanes' z stores happen before lane 0's release
      int old = 0;
      if (lane == 0) old = atomic_add_acq_rel(&st.counters[gi * 8 + rg], 1);
      old = __shfl_sync(0xffffffffu, old, 0);
      if (old == arrivals - 1) {
        if (lane == 0) st.counters[gi * 8 + rg] = 0;  // ready for the next launch
        add_z_planes(st.zws, zplane, st.ks, s_groups.tok + g_begin, g_end - g_begin, st.R_pad, rg * 8, lane);
      }
    }
  }
  if (!ok) {
    if (lane == 0)
      for (int32_t s = 0; s < b.n_sites; ++s) atomicOr(b.site[s].status, EDGELORA_STATUS_TIMEOUT);
    ptx::settle_inline();
  }
}

// ---------------------------------------------------------------------------------------------------------- launch

// The operand ring gets what the other parts leave of an SM's shared memory: the stream of W needs the bytes in flight (28
// sites, 27 tokens: 6 % more with 123 KB per CTA, which leave room for a CTA of the shrink on the same SM, 10 % with
// 104 KB).  Two stages of the expand instead of three: 2 % more.
DecShape decode_sites_shape(int32_t N, int32_t R_pad) {
  DecShape s{};
  const size_t stage = kWBytes + static_cast<size_t>(N) * kBlockK * 2;
  s.exp_bytes = (kTileM * R_pad * 2 + kExpTok * R_pad * 4 + 1023) & ~1023;
  s.exp_stages = 3;
  const size_t fixed = 1024 + kDecTailBytes + static_cast<size_t>(s.exp_stages) * s.exp_bytes;
  s.stages = std::min<int32_t>(kDecMaxStages, static_cast<int32_t>((kDecSmemBudget - fixed) / stage));
  s.smem = fixed + s.stages * stage;
  const int32_t Nc = (N + 31) & ~31;
  s.n_acc = N <= 128 ? 2 : 1;
  s.tmem_cols = 32;
  while (s.tmem_cols < (s.n_acc + 1) * Nc) s.tmem_cols <<= 1;
  return s;
}

cudaError_t decode_sites_set_smem_limit() {
  const int base = static_cast<int>(kDecSmemBudget), shrink = static_cast<int>(kDecShrinkRing + kDecSites * kDecodeMaxT);
  cudaError_t e = cudaSuccess;
#define EDGELORA_SMEM(kernel, bytes) \
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  EDGELORA_SMEM(decode_sites_kernel, base)
  EDGELORA_SMEM(decode_sites_shrink_kernel, shrink)
#undef EDGELORA_SMEM
  return e;
}

cudaError_t launch_decode_sites(const DecBatch &b, const DecShape &shape, int32_t grid, bool pdl, cudaStream_t stream) {
  return launch_ex(decode_sites_kernel, dim3(grid), dim3(kDecThreads), shape.smem, stream, pdl, 1, b);
}
cudaError_t launch_decode_sites_shrink(const DecShrinkBatch &b, int32_t grid, bool pdl, cudaStream_t stream) {
  const size_t ranks = static_cast<size_t>(b.n_sites) * std::min(b.T, b.n_slots);
  return launch_ex(decode_sites_shrink_kernel, dim3(grid), dim3(kDecThreads), kDecShrinkRing + ranks, stream, pdl, 1, b);
}

}  // namespace edgelora
