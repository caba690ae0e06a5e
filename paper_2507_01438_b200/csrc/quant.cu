// Q8_0 adapters (paper Section 5.1: "All LoRA adapters are quantized using the Q8_0 format").
// Q8_0 is the published ggml block format: 32 consecutive values of a row share one half-precision
// scale d and are stored as signed bytes q; the value is d * q.  A block is 34 bytes: d (2 bytes,
// little endian), then q[32].
//
// The kernel here turns an adapter that arrived in this format into the pool's block layout (A padded to [R_pad][h_in], B
// to [h_out][R_pad], bfloat16, padding zero; or A kept in Q8_0, as a plane of bytes and a plane of scales) and writes its
// row of the slot table.  It reads the 8-bit form straight from the page-locked staging buffer: one launch per load, where
// copies of the blocks and of the row around a conversion kernel were four entries on the side stream and twice the
// driver calls, which is what a load cost (two loads in front of a step, 4096 -> 4096, rank 16: 57 us a step, 50 now).
//
#include <cuda_fp16.h>

#include <algorithm>

#include "internal.cuh"
#include "ptx.cuh"

namespace edgelora {

constexpr int kQ8Block = 32;
constexpr int kQ8Bytes = 34;

constexpr int kLoadBlocks = 120;  // Q8_0 blocks of a CTA: 255 pieces of 16 bytes, one per thread
constexpr int kLoadThreads = 256;

struct Q8Load {
  const uint8_t *a, *b;     // page-locked host memory, 16-byte aligned; A_q8 [rank][h_in / 32], B_q8 [h_out][ceil(rank / 32)]
  size_t a_bytes, b_bytes;
  uint16_t *A_blk, *B_blk;  // the slot's blocks
  SlotRow row;              // to *slot when everything else of the slot is on its way too
  SlotRow *slot;
  int32_t R_pad, h_in, h_out, a_ctas, keep_q8;
};

__device__ __forceinline__ uint4 ld_host(const uint8_t *p) {  // (not from a cache that may hold what the buffer held before)
  uint4 v;
  asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// Eight values of a block from its bytes in shared memory, as bfloat16, zero from `n` on (d * q is exact in fp32).
__device__ __forceinline__ uint4 q8_piece(const uint8_t *blk, int piece, int n) {
  const float d = __half2float(__ushort_as_half(*reinterpret_cast<const unsigned short *>(blk)));
  float v[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t w = *reinterpret_cast<const unsigned short *>(blk + 2 + piece * 8 + 2 * i);
    v[2 * i] = 2 * i < n ? d * static_cast<float>(static_cast<int8_t>(w & 255u)) : 0.f;
    v[2 * i + 1] = 2 * i + 1 < n ? d * static_cast<float>(static_cast<int8_t>(w >> 8)) : 0.f;
  }
  return make_uint4(ptx::pack_bf16x2(v[0], v[1]), ptx::pack_bf16x2(v[2], v[3]), ptx::pack_bf16x2(v[4], v[5]),
                    ptx::pack_bf16x2(v[6], v[7]));
}

// The first a_ctas CTAs take 120 blocks of A each (rows from the rank on are zero), the others 120 blocks of B.
__global__ void __launch_bounds__(kLoadThreads) q8_load_kernel(const Q8Load p) {
  __shared__ uint4 s_raw[kLoadBlocks * kQ8Bytes / 16];
  const uint8_t *raw = reinterpret_cast<const uint8_t *>(s_raw);
  const int tid = threadIdx.x;
  const bool is_a = static_cast<int32_t>(blockIdx.x) < p.a_ctas;
  const int32_t chunk = is_a ? blockIdx.x : blockIdx.x - p.a_ctas;
  const uint8_t *from = is_a ? p.a : p.b;
  const size_t at = static_cast<size_t>(chunk) * (kLoadBlocks * kQ8Bytes) + tid * 16, bytes = is_a ? p.a_bytes : p.b_bytes;
  if (tid < kLoadBlocks * kQ8Bytes / 16 && at < bytes)  // (up to 15 bytes behind the end are read: the buffer goes on)
    s_raw[tid] = ld_host(from + at);
  if (blockIdx.x == 0 && tid == 0) *p.slot = p.row;
  __syncthreads();
  const int32_t rank = p.row.rank;
  if (is_a) {
    const int32_t nb = p.h_in / kQ8Block, live = rank * nb, all = p.R_pad * nb;
    for (int i = tid; i < kLoadBlocks * 4; i += kLoadThreads) {
      const int b = i >> 2, piece = i & 3;
      const int32_t block = chunk * kLoadBlocks + b;
      if (block >= all) break;
      const uint8_t *blk = raw + b * kQ8Bytes;
      if (p.keep_q8) {  // bytes [R_pad][h_in], then half-precision scales [R_pad][h_in / 32]
        uint8_t *q = reinterpret_cast<uint8_t *>(p.A_blk);
        uint32_t w[2] = {0u, 0u};
        if (block < live) {
          const unsigned short *h = reinterpret_cast<const unsigned short *>(blk + 2 + piece * 8);
          w[0] = h[0] | static_cast<uint32_t>(h[1]) << 16;
          w[1] = h[2] | static_cast<uint32_t>(h[3]) << 16;
        }
        *reinterpret_cast<uint2 *>(q + static_cast<size_t>(block) * kQ8Block + piece * 8) = make_uint2(w[0], w[1]);
        if (piece == 0)
          reinterpret_cast<unsigned short *>(q + static_cast<size_t>(all) * kQ8Block)[block] =
              block < live ? *reinterpret_cast<const unsigned short *>(blk) : static_cast<unsigned short>(0);
      } else {
        *reinterpret_cast<uint4 *>(p.A_blk + static_cast<size_t>(block) * kQ8Block + piece * 8) =
            block < live ? q8_piece(blk, piece, 8) : make_uint4(0u, 0u, 0u, 0u);
      }
    }
  } else {
    const int32_t nb = (rank + kQ8Block - 1) / kQ8Block, rows = kLoadBlocks / nb, pieces = p.R_pad >> 3;
    const int32_t j0 = chunk * rows, n = min(rows, p.h_out - j0) * pieces;
    for (int i = tid; i < n; i += kLoadThreads) {
      const int32_t r = i / pieces, c = (i - r * pieces) * 8;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (c < rank) v = q8_piece(raw + (r * nb + c / kQ8Block) * kQ8Bytes, (c & (kQ8Block - 1)) >> 3, rank - c);
      *reinterpret_cast<uint4 *>(p.B_blk + static_cast<size_t>(j0 + r) * p.R_pad + c) = v;
    }
  }
}

// Base weights stored in a block format (paper Section 5.1, model table: base models in Q8_0 or
// Q4_0).  Q4_0 is the published ggml format of 18 bytes per 32 consecutive values of a row: a
// half-precision scale d, then 16 bytes; byte j holds value j in its low four bits and value j + 16
// in its high four bits, each as an unsigned code c with value d * (c - 8).  One thread decodes one
// block into 32 bfloat16 values (round to nearest even; d * code is exact in fp32).
template <int kFormat>  // 0: Q8_0, 1: Q4_0
__global__ void __launch_bounds__(256)
weights_decode_kernel(const uint8_t *__restrict__ Wq, uint16_t *__restrict__ W, size_t n_blocks) {
  constexpr int kBytes = kFormat == 0 ? kQ8Bytes : 18;
  for (size_t b = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; b < n_blocks;
       b += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const uint8_t *blk = Wq + b * kBytes;
    const float d = __half2float(__ushort_as_half(static_cast<unsigned short>(blk[0] | (blk[1] << 8))));
    float v[32];
    if (kFormat == 0) {
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = d * static_cast<float>(static_cast<int8_t>(blk[2 + i]));
    } else {
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int byte = blk[2 + j];
        v[j] = d * static_cast<float>((byte & 0xF) - 8);
        v[j + 16] = d * static_cast<float>((byte >> 4) - 8);
      }
    }
    uint4 *dst = reinterpret_cast<uint4 *>(W + b * 32);  // blocks follow one another along the rows
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint4 o;
      o.x = ptx::pack_bf16x2(v[8 * q + 0], v[8 * q + 1]);
      o.y = ptx::pack_bf16x2(v[8 * q + 2], v[8 * q + 3]);
      o.z = ptx::pack_bf16x2(v[8 * q + 4], v[8 * q + 5]);
      o.w = ptx::pack_bf16x2(v[8 * q + 6], v[8 * q + 7]);
      dst[q] = o;
    }
  }
}

cudaError_t launch_weights_decode(int32_t format, const uint8_t *Wq, uint16_t *W, size_t n_blocks, cudaStream_t stream) {
  const int grid = static_cast<int>(std::min<size_t>((n_blocks + 255) / 256, 148 * 8));
  if (format == 0)
    weights_decode_kernel<0><<<grid, 256, 0, stream>>>(Wq, W, n_blocks);
  else
    weights_decode_kernel<1><<<grid, 256, 0, stream>>>(Wq, W, n_blocks);
  return cudaGetLastError();
}

cudaError_t launch_q8_load(const uint8_t *a_pinned, size_t a_bytes, const uint8_t *b_pinned, size_t b_bytes, uint16_t *A_blk,
                           uint16_t *B_blk, const SlotRow &row, SlotRow *slot, int32_t R_pad, int32_t h_in, int32_t h_out,
                           bool keep_q8, cudaStream_t stream) {
  const int32_t a_ctas = (R_pad * (h_in / kQ8Block) + kLoadBlocks - 1) / kLoadBlocks;
  const int32_t rows = kLoadBlocks / ((row.rank + kQ8Block - 1) / kQ8Block), b_ctas = (h_out + rows - 1) / rows;
  const Q8Load p{a_pinned, b_pinned, a_bytes, b_bytes, A_blk, B_blk, row, slot, R_pad, h_in, h_out, a_ctas, keep_q8 ? 1 : 0};
  q8_load_kernel<<<a_ctas + b_ctas, kLoadThreads, 0, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace edgelora

extern "C" int edgelora_weights_decode(int32_t format, const void *W_blocks_dev, int32_t h_out, int32_t h_in,
                                       uint16_t *W_dev, void *stream) {
  if ((format != EDGELORA_WEIGHTS_Q8_0 && format != EDGELORA_WEIGHTS_Q4_0) || !W_blocks_dev || !W_dev || h_out <= 0 ||
      h_in <= 0 || h_in % 32 != 0)
    return EDGELORA_ERR_INVALID_ARG;
  const size_t n_blocks = static_cast<size_t>(h_out) * (h_in / 32);
  const cudaError_t e = edgelora::launch_weights_decode(format, static_cast<const uint8_t *>(W_blocks_dev), W_dev, n_blocks,
                                                        static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) {
    edgelora::set_last_cuda_error(e, "weights_decode_kernel");
    return EDGELORA_ERR_CUDA;
  }
  return EDGELORA_OK;
}
