// The low-rank intermediate of a token as the bf16 operand of the expand (shared by the kernels that write it
// and the kernels that add B_a z on the tensor cores).
#pragma once
#include "internal.cuh"
#include "ptx.cuh"

namespace edgelora {

// Eight consecutive values of z as one 16-byte chunk of the operand: the zsplits partial planes (`plane` floats
// apart) are added in order, values at or past the true rank forced to zero.  z: the first of the eight in plane 0,
// r0: its rank index.
__device__ __forceinline__ uint4 z_chunk(const float *z, size_t plane, int32_t zsplits, int32_t r0, int32_t rank) {
  float acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.f;
#pragma unroll 8
  for (int sp = 0; sp < zsplits; ++sp) {
    const float4 *zp = reinterpret_cast<const float4 *>(z + sp * plane);
    const float4 u = __ldcg(zp), w = __ldcg(zp + 1);
    acc[0] += u.x; acc[1] += u.y; acc[2] += u.z; acc[3] += u.w;
    acc[4] += w.x; acc[5] += w.y; acc[6] += w.z; acc[7] += w.w;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (r0 + i >= rank) acc[i] = 0.f;
  return make_uint4(ptx::pack_bf16x2(acc[0], acc[1]), ptx::pack_bf16x2(acc[2], acc[3]), ptx::pack_bf16x2(acc[4], acc[5]),
                    ptx::pack_bf16x2(acc[6], acc[7]));
}

// z of token t from one summed fp32 plane [max_tokens][R_pad] as packed bf16 (eight 16-byte chunks; chunks at or
// past the rank stride are zero).
__device__ __forceinline__ void load_z_packed(const float *zws, int32_t R_pad, int32_t max_tokens, uint32_t *status,
                                              int32_t t, int32_t rank, uint4 (&out)[8]) {
  if (!EL_CHECK(status, rank <= R_pad && t >= 0 && t < max_tokens, 3)) {
    rank = 0;  // all zeros, read from row 0
    t = 0;
  }
  const int nch = R_pad >> 3;
#pragma unroll
  for (int c = 0; c < 8; ++c)
    out[c] = c < nch ? z_chunk(zws + static_cast<size_t>(t) * R_pad + c * 8, 0, 1, c * 8, rank)
                     : make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace edgelora
