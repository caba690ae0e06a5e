// The expand on the CUDA cores, as the decode kernels share it: rows of B_a in shared memory against fp32 z (paper Section
// 2.1 for B: h_out x r).
#pragma once
#include "internal.cuh"
#include "ptx.cuh"

namespace edgelora {

// How the 16-byte chunks of row `row` are swizzled in a tiled copy whose rows are R_pad * 2 = 32, 64 or 128 bytes long: chunk
// c lies at c ^ this.
__device__ __forceinline__ int row_swizzle(int row, int R_pad) {
  return R_pad == 64 ? row & 7 : R_pad == 32 ? (row >> 1) & 3 : (row >> 2) & 1;
}

// A row of B_a (its 16-byte chunks swizzled by `sw`) against the z rows of kTok tokens, z_bytes apart: the first kChunks groups
// of eight rank rows.  What bounds a stage is the latency of this chain, in a single warp per scheduler: so no branches (they
// kept the loads of a chunk behind the sums of the one before it, 75 cycles a chunk and token), and two sums of two values per
// token; with many tokens it is the reads of shared memory.  So the callers take the form that ends at the adapter's rank, not at
// the pool's stride (680 -> 9576, 97 tokens on seven adapters of rank 16 to 64, stride 64: 31.6 us per call, now 27.7; 472 -> 12488,
// 177 on 24: 44.0 and 36.6).  z is read up to the last live group of eight rank rows; what lies behind it was not written.
template <int kChunks, int kTok>
__device__ __forceinline__ void expand_dots(const uint8_t *brow, int sw, uint32_t z, uint32_t z_bytes, int rank, float *acc) {
  uint64_t s0[kTok], s1[kTok];
#pragma unroll
  for (int q = 0; q < kTok; ++q) s0[q] = s1[q] = 0;
#pragma unroll
  for (int c = 0; c < kChunks; ++c) {
    const uint32_t live = c * 8 < rank ? 1u : 0u;
    const uint4 bb = *reinterpret_cast<const uint4 *>(brow + ((c ^ sw) << 4));
    uint64_t u[kTok][4];
#pragma unroll
    for (int q = 0; q < kTok; ++q) {
      ptx::ld_shared_f32x4_if(z + q * z_bytes + c * 32, live, u[q][0], u[q][1]);
      ptx::ld_shared_f32x4_if(z + q * z_bytes + c * 32 + 16, live, u[q][2], u[q][3]);
    }
    const uint64_t f0 = ptx::f32x2(ptx::bf16_lo(bb.x), ptx::bf16_hi(bb.x)), f1 = ptx::f32x2(ptx::bf16_lo(bb.y), ptx::bf16_hi(bb.y));
    const uint64_t f2 = ptx::f32x2(ptx::bf16_lo(bb.z), ptx::bf16_hi(bb.z)), f3 = ptx::f32x2(ptx::bf16_lo(bb.w), ptx::bf16_hi(bb.w));
#pragma unroll
    for (int q = 0; q < kTok; ++q) {
      s0[q] = ptx::fma_f32x2(f0, u[q][0], s0[q]);
      s1[q] = ptx::fma_f32x2(f1, u[q][1], s1[q]);
      s0[q] = ptx::fma_f32x2(f2, u[q][2], s0[q]);
      s1[q] = ptx::fma_f32x2(f3, u[q][3], s1[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < kTok; ++q) acc[q] = ptx::sum_f32x2(s0[q], s1[q]);
}

}  // namespace edgelora
