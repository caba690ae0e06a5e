// Scoring head of the adapter router (paper Section 3.2: one score in [0, 1] per adapter for a
// prompt; Section 5.1: a classification head on the base model): scores[b][j] =
// sigmoid(W_r[j] . h[b] + bias[j]).  One pass over W_r ([n][hidden] bf16, 8-16 MB for the paper's
// 1000-2000 adapters) is all the memory traffic there is; what bounds a launch of a few
// microseconds is the chain of its latencies: the first round trip to HBM, the dot products of a
// warp, the sums over lanes and warps.  fp32 accumulation, fp32 scores.
#include "internal.cuh"
#include "launch.cuh"
#include "ptx.cuh"

namespace edgelora {

constexpr int kRouterMaxHidden = 8192;
constexpr int kRouterRows = 8;      // rows of W_r of a CTA
constexpr int kRouterPrompts = 8;   // prompts of a pass: the n of the matrix instruction

// Without overflow on either side.
__device__ __forceinline__ float sigmoid(float v) {
  const float e = __expf(-fabsf(v));
  return v >= 0.f ? 1.f / (1.f + e) : e / (1.f + e);
}

// D[16 x 8] = A[16 x 16] * B[16 x 8] for rows 0..7 of A and D (the others are zero).  Lane 4 g + t holds of A and B the
// values {2 t, 2 t + 1} (a0, b0) and {2 t + 8, 2 t + 9} (a1, b1) of row g, and of D row g, columns 2 t and 2 t + 1.
__device__ __forceinline__ void mma_rows8(float &d0, float &d1, uint32_t a0, uint32_t a1, uint32_t b0, uint32_t b1) {
  float z0 = 0.f, z1 = 0.f;
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %5}, {%7, %8}, {%0, %1, %2, %3};"
      : "+f"(d0), "+f"(d1), "+f"(z0), "+f"(z1)
      : "r"(a0), "r"(0u), "r"(a1), "r"(b0), "r"(b1));
}

// A CTA takes eight rows of W_r, each of its kWarps warps an equal part of their values, and requests all of it at once: with the rows
// of W_r spread over the warps of the chip, all of it is in flight in one round.  The products run on the warp-level matrix
// instruction, whose operands are registers: the sum over k may be taken in any order, so lane 4 g + t takes 16 bytes of
// row g of W_r and of prompt g as they lie in memory, and no value is moved or converted.  (A tile of the tcgen05 pipe is
// 128 rows: eight of them for 1000 adapters.  On the CUDA cores a prompt cost 1.1 us for 1000 x 4096.)  The
// instruction sums 16 products; everything beyond that is added in fp32, in a tree (with the chunks summed one after the
// other the scores were up to 8.0e-8 of their norm away from the same sums in 64 bits, 6.9e-8 on the CUDA cores).
// Us per call, CUDA graph over three copies of W_r, a warp per row on the CUDA cores (router_rows_kernel) and here: 1000 x 4096,
// 4 / 16 prompts: 6.8 / 21.9 and 3.7 / 6.1; 200 x 2048, 16 prompts: 16.1 and 4.1; 2000 x 8192, 3 / 16 prompts: 12.8 / 81.8
// and 9.5 / 16.0.
template <int kWarps>
__global__ void __launch_bounds__(kWarps * 32, 16 / kWarps)
router_scores_kernel(const uint16_t *__restrict__ Wr, const float *__restrict__ bias,
                     const uint16_t *__restrict__ h, int32_t B, int32_t n, int32_t hidden,
                     float *__restrict__ scores) {
  __shared__ float s_sum[kWarps][kRouterRows][kRouterPrompts];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int n8 = hidden >> 3, n_chunks = (n8 + 3) >> 2;  // 16-byte pieces and chunks of a row
  const int per = (n_chunks + kWarps - 1) / kWarps, c_begin = warp * per, c_end = min(n_chunks, c_begin + per);
  const int j0 = blockIdx.x * kRouterRows;
  const uint4 *row = reinterpret_cast<const uint4 *>(Wr + static_cast<size_t>(min(j0 + g, n - 1)) * hidden);
  ptx::pdl_launch_dependents();
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  auto load8 = [&](const uint4 *from, int c0, uint4 (&v)[8]) {  // this lane's pieces of the chunks from c0 on
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = (c0 + u) * 4 + t;
      v[u] = c0 + u < c_end && k < n8 ? __ldg(from + k) : zero;
    }
  };
  uint4 w0[8], w1[8];  // 16 chunks: all of a warp's part of rows up to 4096 values long
  load8(row, c_begin, w0);
  load8(row, c_begin + 8, w1);
  ptx::pdl_wait_prior_grids();  // h comes from earlier work on the stream
#pragma unroll 1
  for (int b0 = 0; b0 < B; b0 += kRouterPrompts) {
    const uint4 *prompt = reinterpret_cast<const uint4 *>(h + static_cast<size_t>(min(b0 + g, B - 1)) * hidden);
    float s0 = 0.f, s1 = 0.f;
    auto add8 = [&](int c0, const uint4 (&w)[8]) {
      uint4 x[8];
      load8(prompt, c0, x);
#pragma unroll
      for (int u0 = 0; u0 < 8; u0 += 4) {
        float d0[8], d1[8];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          d0[2 * u] = d1[2 * u] = d0[2 * u + 1] = d1[2 * u + 1] = 0.f;
          mma_rows8(d0[2 * u], d1[2 * u], w[u0 + u].x, w[u0 + u].y, x[u0 + u].x, x[u0 + u].y);
          mma_rows8(d0[2 * u + 1], d1[2 * u + 1], w[u0 + u].z, w[u0 + u].w, x[u0 + u].z, x[u0 + u].w);
        }
#pragma unroll
        for (int m = 4; m >= 1; m >>= 1)
#pragma unroll
          for (int u = 0; u < m; ++u) {
            d0[u] += d0[u + m];
            d1[u] += d1[u + m];
          }
        s0 += d0[0];
        s1 += d1[0];
      }
    };
#pragma unroll 1
    for (int c = c_begin; c < c_end; c += 16) {
      // longer rows: the chunks 16 further on, or at the end those that the next prompts begin with, follow into the
      // registers that a half of the 16 leaves
      const int next = c + 16 < c_end ? c + 16 : b0 + kRouterPrompts < B ? c_begin : -1;
      const bool more = per > 16 && next >= 0;
      add8(c, w0);
      if (more) load8(row, next, w0);
      if (c + 8 < c_end) add8(c + 8, w1);
      if (more) load8(row, next + 8, w1);
    }
    s_sum[warp][g][2 * t] = s0;
    s_sum[warp][g][2 * t + 1] = s1;
    __syncthreads();
    if (threadIdx.x < kRouterRows * kRouterPrompts) {  // a thread per score
      const int r = threadIdx.x & 7, q = threadIdx.x >> 3, j = j0 + r;
      if (j < n && b0 + q < B) {
        float part[kWarps];
#pragma unroll
        for (int p = 0; p < kWarps; ++p) part[p] = s_sum[p][r][q];
#pragma unroll
        for (int m = kWarps / 2; m >= 1; m >>= 1)
#pragma unroll
          for (int p = 0; p < m; ++p) part[p] += part[p + m];
        float v = part[0];
        if (bias) v += bias[j];
        scores[static_cast<size_t>(b0 + q) * n + j] = sigmoid(v);
      }
    }
    __syncthreads();  // s_sum is written again
  }
}

// A warp owns a row of W_r and asks for (the first 8 KB of) its first one, 512 contiguous bytes per load, before the prompts are
// staged in shared memory; dot products on the CUDA cores, lanes added by shuffles.  What bounds it is the first round trip to
// HBM and then 1.1 us for every prompt of 1000 x 4096, so it is launched for a single one.  The loops over prompts are rolled, also
// for that one: with their count known to the compiler the call is 0.1 to 0.3 us longer.
constexpr int kRowThreads = 256;
constexpr int kRowPrompts = 8;  // prompts per pass over a row
constexpr int kRowUnroll = 16;  // 16-byte loads per lane in flight: a whole row of 4096 values
__global__ void __launch_bounds__(kRowThreads)
router_rows_kernel(const uint16_t *__restrict__ Wr, const float *__restrict__ bias, const uint16_t *__restrict__ h,
                   int32_t B, int32_t n, int32_t hidden, float *__restrict__ scores) {
  extern __shared__ uint4 s_h[];  // [min(B, 8)][hidden / 8]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n8 = hidden >> 3;
  const int j_first = blockIdx.x * (kRowThreads / 32) + warp, j_step = gridDim.x * (kRowThreads / 32);
  ptx::pdl_launch_dependents();
  auto load_chunk = [&](int j, int k0, uint4 (&wv)[kRowUnroll]) {
    const uint4 *row = reinterpret_cast<const uint4 *>(Wr + static_cast<size_t>(j) * hidden);
#pragma unroll
    for (int u = 0; u < kRowUnroll; ++u)
      wv[u] = (k0 + 32 * u < n8) ? __ldg(row + k0 + 32 * u) : make_uint4(0u, 0u, 0u, 0u);
  };
  uint4 wv[kRowUnroll];
  if (j_first < n) load_chunk(j_first, lane, wv);  // W_r is not written by anything on the stream
  ptx::pdl_wait_prior_grids();                      // h comes from earlier work on the stream
  for (int b0 = 0; b0 < B; b0 += kRowPrompts) {
    const int nb = min(kRowPrompts, B - b0);
    __syncthreads();
    for (int i = threadIdx.x; i < nb * n8; i += kRowThreads)
      s_h[i] = __ldg(reinterpret_cast<const uint4 *>(h + static_cast<size_t>(b0) * hidden) + i);
    __syncthreads();
    for (int j = j_first; j < n; j += j_step) {
      float v = 0.f;  // lane q: W_r[j] . h[b0 + q]
      for (int k0 = lane; k0 < n8; k0 += 32 * kRowUnroll) {
        if (!(b0 == 0 && j == j_first && k0 == lane)) load_chunk(j, k0, wv);  // the first chunk is already here
#pragma unroll 1
        for (int q = 0; q < nb; ++q) {
          const uint4 *hq = s_h + q * n8 + k0;
          float s = 0.f;
#pragma unroll
          for (int u = 0; u < kRowUnroll; ++u) {
            if (k0 + 32 * u < n8) {  // (values past the row are zero: nothing to add)
              const uint4 w = wv[u], x = hq[32 * u];
              s = fmaf(ptx::bf16_lo(w.x), ptx::bf16_lo(x.x), s); s = fmaf(ptx::bf16_hi(w.x), ptx::bf16_hi(x.x), s);
              s = fmaf(ptx::bf16_lo(w.y), ptx::bf16_lo(x.y), s); s = fmaf(ptx::bf16_hi(w.y), ptx::bf16_hi(x.y), s);
              s = fmaf(ptx::bf16_lo(w.z), ptx::bf16_lo(x.z), s); s = fmaf(ptx::bf16_hi(w.z), ptx::bf16_hi(x.z), s);
              s = fmaf(ptx::bf16_lo(w.w), ptx::bf16_lo(x.w), s); s = fmaf(ptx::bf16_hi(w.w), ptx::bf16_hi(x.w), s);
            }
          }
#pragma unroll
          for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
          if (lane == q) v += s;
        }
      }
      if (lane < nb) {
        if (bias) v += bias[j];
        scores[static_cast<size_t>(b0 + lane) * n + j] = sigmoid(v);
      }
    }
  }
}

}  // namespace edgelora

extern "C" int edgelora_router_scores(const void *Wr_dev, const float *bias_dev, const void *h_dev, int32_t B,
                                      int32_t n, int32_t hidden, float *scores_dev, void *stream) {
  using namespace edgelora;
  if (B < 0 || n < 1 || hidden < 8 || (hidden & 7) || hidden > kRouterMaxHidden) return EDGELORA_ERR_INVALID_ARG;
  if (B == 0) return EDGELORA_OK;
  if (!Wr_dev || !h_dev || !scores_dev) return EDGELORA_ERR_INVALID_ARG;
  // Eight warps hold rows of 4096 values in their registers at once, two CTAs to an SM; longer rows are better off with
  // sixteen, as long as every CTA has an SM (1000 x 8192, one prompt: 4.7 us against 5.6; 2000 x 8192: 10.1 against 9.0).
  const int grid = (n + kRouterRows - 1) / kRouterRows;
  auto launch = [&](auto kernel, int warps) {
    return launch_ex(kernel, dim3(grid), dim3(warps * 32), 0, static_cast<cudaStream_t>(stream), false, 1,
                     static_cast<const uint16_t *>(Wr_dev), bias_dev, static_cast<const uint16_t *>(h_dev), B, n, hidden,
                     scores_dev);
  };
  const bool wide = hidden > 4096 && grid <= 128;
  // A single prompt: a warp per row, but for rows of at most 2048 values and those that sixteen warps share.  Us per call with
  // W_r in L2 and, in brackets, out of HBM, on the matrix instruction and a warp per row: 200 x 4096: 3.64 and 3.36; 1000 x
  // 4096: 3.76 (4.68) and 3.48 (4.68); 2000 x 4096: 4.67 (6.07) and 4.39 (6.16); 1200 x 8192: 7.2 (9.1) and 6.2 (8.3); 2000 x
  // 8192: 9.1 (9.9) and 7.5 (9.8).  1000 x 2048: 3.07 with either; 1000 x 8192, sixteen warps: 4.9 (6.3) and 5.3 (7.7).
  const bool one = B == 1 && hidden > 2048 && !wide;
  cudaError_t e;
  if (one)
    e = launch_ex(router_rows_kernel, dim3((n + kRowThreads / 32 - 1) / (kRowThreads / 32)), dim3(kRowThreads),
                  static_cast<size_t>(hidden) * 2, static_cast<cudaStream_t>(stream), false, 1,
                  static_cast<const uint16_t *>(Wr_dev), bias_dev, static_cast<const uint16_t *>(h_dev), B, n, hidden, scores_dev);
  else
    e = wide ? launch(router_scores_kernel<16>, 16) : launch(router_scores_kernel<8>, 8);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return EDGELORA_ERR_CUDA;
  }
  return EDGELORA_OK;
}
