// Eight rows of A against up to four rows of x by one warp, streamed through the warp's own ring in shared memory (the
// inner part of the decode shrinks).
#pragma once
#include <cuda_fp16.h>

#include "internal.cuh"
#include "ptx.cuh"

namespace edgelora {

constexpr int kDsTok = kDecShrinkTok;

__device__ __forceinline__ void unpack8(const uint4 &v, float (&f)[8]) {
  f[0] = ptx::bf16_lo(v.x); f[1] = ptx::bf16_hi(v.x);
  f[2] = ptx::bf16_lo(v.y); f[3] = ptx::bf16_hi(v.y);
  f[4] = ptx::bf16_lo(v.z); f[5] = ptx::bf16_hi(v.z);
  f[6] = ptx::bf16_lo(v.w); f[7] = ptx::bf16_hi(v.w);
}

constexpr int kDsMaxDepth = 5;                      // ring stages per warp: up to 5, or 2 for small batches
constexpr int kDsRowBytes = kShrinkStepElems * 2;   // 512: one row segment of one K step
constexpr int kDsStageBytes = (8 + kDsTok) * kDsRowBytes;  // 8 rows of A, then up to 4 rows of x

// Eight rows of A against NT token rows of x over the K steps [step0, step1).  One K step is 256
// elements; lane l owns elements [8 l, 8 l + 8) of it.  The warp's lane 0 keeps kDsDepth - 1 steps
// in flight with TMA copies (one box of 8 x 512 bytes of A and one 512-byte row of x per token)
// into the warp's private ring; columns past h_in arrive as zeros.  `phase` holds one parity bit
// per ring stage and lives across calls.  Returns false if a wait gave up.
// The ring's bytes are those of kDsDepth stages with four x rows; with fewer x rows a stage is
// shorter, and with one token five stages fit where four did: a third more bytes in flight for the
// items that dominate a many-adapter batch (the stream is bound by latency times bytes in flight).
template <int NT, int kDsDepth>
struct RingShape {
  static constexpr int kStage = (8 + NT) * kDsRowBytes;
  static constexpr int kDepth = (kDsDepth * kDsStageBytes) / kStage > kDsMaxDepth ? kDsMaxDepth
                                                                                  : (kDsDepth * kDsStageBytes) / kStage;
};
// kQ8: the A rows are kept in Q8_0 (paper Section 5.1: per 32 values a half-precision scale d and 32
// signed bytes q, value d * q), in the pool as two planes per slot: the bytes [R_pad][h_in] and the
// scales [R_pad][h_in / 32].  A K step of 256 values is then 256 bytes + 8 scales per row: two boxes
// per step (8 x 256 bytes at the start of the stage, 8 x 16 bytes behind them), and lane l decodes the
// eight values it owns (one aligned 8-byte load, block l / 4) on the fly: sum_e q_e x_e in fp32,
// times d once.  17/32 of the bytes of the bfloat16 rows.
constexpr int kQ8QBytes = kShrinkStepElems;            // 256 bytes of q per row and step
constexpr int kQ8DBytes = (kShrinkStepElems / 32) * 2;  // 16 bytes of scales per row and step
// signed byte i of w as a float: the byte with its sign bit flipped is q + 128, placed in the
// mantissa of 2^23 it reads 2^23 + 128 + q
__device__ __forceinline__ float s8_to_float(uint32_t w_flipped, int i) {
  return __uint_as_float(__byte_perm(w_flipped, 0x4B000000u, 0x7440u + i)) - 8388736.0f;
}
template <int NT, int kDsDepthCfg, bool kQ8>
__device__ __forceinline__ bool shrink_rows8(const CUtensorMap *tmap_a, const CUtensorMap *tmap_d,
                                             const CUtensorMap *tmap_x,
                                             int32_t slot, int32_t row0, const int32_t (&tok)[kDsTok],
                                             int step0, int step1, int stride, uint8_t *ring, uint64_t *bars,
                                             uint32_t &phase, int lane, float (&acc)[8 * kDsTok]) {
  constexpr int kDsDepth = RingShape<NT, kDsDepthCfg>::kDepth;
  constexpr int kStage = RingShape<NT, kDsDepthCfg>::kStage;
  auto issue = [&](int step, int stage) {
    if (step < step1 && ptx::elect_one()) {
      uint8_t *dst = ring + stage * kStage;
      ptx::mbar_arrive_expect_tx_relaxed(&bars[stage],
                                         (kQ8 ? 8 * (kQ8QBytes + kQ8DBytes) : 8 * kDsRowBytes) + NT * kDsRowBytes);
      ptx::tma_load_3d(dst, tmap_a, &bars[stage], step * (kQ8 ? kQ8QBytes / 2 : kShrinkStepElems), row0, slot);
      if (kQ8) ptx::tma_load_3d(dst + 8 * kQ8QBytes, tmap_d, &bars[stage], step * (kShrinkStepElems / 32), row0, slot);
#pragma unroll
      for (int q = 0; q < NT; ++q)
        ptx::tma_load_2d(dst + (8 + q) * kDsRowBytes, tmap_x, &bars[stage], step * kShrinkStepElems, tok[q]);
    }
  };
#pragma unroll
  for (int d = 0; d < kDsDepth - 1; ++d) issue(step0 + d * stride, d);
  int stage = 0;
  for (int step = step0; step < step1; step += stride) {
    __syncwarp();  // every lane has finished reading the stage that is refilled next
    issue(step + (kDsDepth - 1) * stride, (stage + kDsDepth - 1) % kDsDepth);
    if (!ptx::mbar_wait(&bars[stage], (phase >> stage) & 1u)) return false;
    phase ^= 1u << stage;
    const uint4 *src = reinterpret_cast<const uint4 *>(ring + stage * kStage) + lane;
    float xf[NT][8];
#pragma unroll
    for (int q = 0; q < NT; ++q) unpack8(src[(8 + q) * (kDsRowBytes / 16)], xf[q]);
    if (kQ8) {
      const uint8_t *st = ring + stage * kStage;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const uint2 qq = *reinterpret_cast<const uint2 *>(st + r * kQ8QBytes + lane * 8);
        const float d = __half2float(__ushort_as_half(
            *reinterpret_cast<const unsigned short *>(st + 8 * kQ8QBytes + r * kQ8DBytes + (lane >> 2) * 2)));
        const uint32_t w0 = qq.x ^ 0x80808080u, w1 = qq.y ^ 0x80808080u;
        float qf[8];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          qf[e] = s8_to_float(w0, e);
          qf[4 + e] = s8_to_float(w1, e);
        }
#pragma unroll
        for (int q = 0; q < NT; ++q) {
          float part = 0.f;
#pragma unroll
          for (int e = 0; e < 8; ++e) part = fmaf(qf[e], xf[q][e], part);
          acc[r * kDsTok + q] = fmaf(d, part, acc[r * kDsTok + q]);
        }
      }
    } else {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        float af[8];
        unpack8(src[r * (kDsRowBytes / 16)], af);
#pragma unroll
        for (int q = 0; q < NT; ++q)
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[r * kDsTok + q] = fmaf(af[e], xf[q][e], acc[r * kDsTok + q]);
      }
    }
    if (++stage == kDsDepth) stage = 0;
  }
  return true;
}

// The sums over the warp's lanes of 32 values at once: lane L ends with that of value L, in acc[0].
__device__ __forceinline__ void sum_over_lanes(float (&acc)[8 * kDsTok], int lane) {
#pragma unroll
  for (int off = 16, cnt = 16; off >= 1; off >>= 1, cnt >>= 1) {
    const bool upper = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < cnt; ++i) {
      const float send = upper ? acc[i] : acc[i + cnt];
      const float keep = upper ? acc[i + cnt] : acc[i];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
}

// The K chunks' partial planes added in order into the plane that the expand reads, by one warp: eight rank rows from r0 on of
// the n tokens `tok` of an adapter.  What bounds it is the latency of a round of loads, behind everything else of the launch:
// 16 planes of up to four tokens in one round, four planes of 16 tokens where an adapter has more of them.  (A token's planes are
// added by the last warp of its adapter alone, so an adapter with many tokens is what the launch ends on.  Four tokens in a
// round whatever their number, and now, us per call: 4616 -> 4136, 225 tokens on seven adapters: 49.0 and 40.9; 2584 -> 3264, 158
// on four: 47.4 and 41.4; 1848 -> 288, 255 on 56: 35.7 and 31.4; 14336 -> 4096, 256 on about 100: 87.1 and 85.8.)
__device__ __forceinline__ void add_z_planes(float *zws, size_t zplane, int ks, const uint8_t *tok, int n, int R_pad, int r0,
                                             int lane) {
  if (n <= 4) {
    if (lane >= n * 8) return;
    const size_t off = static_cast<size_t>(tok[lane >> 3]) * R_pad + r0 + (lane & 7);
    float part[kMaxZSplits];
#pragma unroll
    for (int sp = 0; sp < kMaxZSplits; ++sp) part[sp] = sp < ks ? __ldcg(zws + sp * zplane + off) : 0.f;
    float sum = 0.f;
#pragma unroll
    for (int sp = 0; sp < kMaxZSplits; ++sp) sum += part[sp];
    zws[kMaxZSplits * zplane + off] = sum;
    return;
  }
#pragma unroll 1
  for (int i0 = lane; i0 < n * 8; i0 += 128) {
    size_t off[4];
    float sum[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      off[e] = static_cast<size_t>(tok[min(i0 + 32 * e, n * 8 - 1) >> 3]) * R_pad + r0 + (lane & 7);
      sum[e] = 0.f;
    }
#pragma unroll 1
    for (int s0 = 0; s0 < ks; s0 += 4) {
      float part[4][4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int e = 0; e < 4; ++e) part[k][e] = s0 + k < ks ? __ldcg(zws + (s0 + k) * zplane + off[e]) : 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int e = 0; e < 4; ++e) sum[e] += part[k][e];
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (i0 + 32 * e < n * 8) zws[kMaxZSplits * zplane + off[e]] = sum[e];
  }
}

__device__ __forceinline__ int atomic_add_acq_rel(int32_t *p, int v) {
  int old;
  asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}

}  // namespace edgelora
