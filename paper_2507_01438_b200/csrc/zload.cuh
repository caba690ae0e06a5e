// The low-rank intermediate of a token as the bf16 operand of the expand (shared by the kernels that write it
// and the kernels that add B_a z on the tensor cores).
#pragma once
#include "internal.cuh"
#include "ptx.cuh"

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

// z of token t from one summed fp32 plane [max_tokens][R_pad] as packed bf16 (eight 16-byte chunks; chunks at or
// past the rank stride are zero).
__device__ __forceinline__ void load_z_packed(const float *zws, int32_t R_pad, int32_t max_tokens, uint32_t *status,
                                              int32_t t, int32_t rank, uint4 (&out)[8]) {
  if (!EL_CHECK(status, rank <= R_pad && t >= 0 && t < max_tokens, 3)) {
    rank = 0;  // all zeros, read from row 0
    t = 0;
  }
  const int nch = R_pad >> 3;
  const float4 *zt = reinterpret_cast<const float4 *>(zws + static_cast<size_t>(t) * R_pad);
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    out[c] = make_uint4(0u, 0u, 0u, 0u);
    if (c < nch) {
      const float4 u = __ldcg(zt + 2 * c), w = __ldcg(zt + 2 * c + 1);
      const float v[8] = {u.x, u.y, u.z, u.w, w.x, w.y, w.z, w.w};
      out[c] = pack_z_chunk(v, c * 8, rank);
    }
  }
}

}  // namespace edgelora
