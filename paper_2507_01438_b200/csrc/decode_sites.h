// What the kernels of decode_sites.cu are launched with: a run of linear sites over one decode-sized batch.
#pragma once
#include "internal.cuh"

namespace edgelora {

constexpr int kDecSites = 32;   // sites of one launch at most
constexpr int kDecInputs = 4;   // distinct inputs of one launch at most
constexpr int kDecThreads = 256;
constexpr int kDecMaxStages = 12;
constexpr int kDecMaxExpStages = 4;
constexpr size_t kDecTailBytes = 8192;

struct DecSite {
  CUtensorMap w;         // W [h_out][h_in], boxes of 128 rows x 64
  CUtensorMap b;         // the pool's B blocks [S][h_out][R_pad], boxes of 128 rows x R_pad
  uint16_t *y;           // [T][h_out]
  const SlotRow *slots;
  const float *z;        // [max_tokens][R_pad], live groups of eight rank rows only
  uint32_t *status;
  int32_t x_index, h_out, kb, R_pad;
};
struct DecBatch {
  CUtensorMap x[kDecInputs];  // [T][h_in], boxes of N rows x 64
  DecSite site[kDecSites];
  int32_t n_sites, T, n_slots;
  int32_t N;             // UMMA N: tokens rounded up to 16
  int32_t stages, exp_stages, exp_bytes;  // operand ring, expand ring and the bytes of one of its stages
  int32_t n_acc, tmem_cols;
  const int32_t *ids;    // the caller's ids (validated again inside the kernel)
  float *partial;        // two planes [N][128] per CTA: of the first and of the last piece of its run
  int32_t *arrivals;     // [CTAs][4]: by the CTA in whose run the tile begins, zero in front of the launch
  long long wait_cycles;
};

struct DecShrinkSite {
  CUtensorMap a;         // the pool's A blocks [S][R_pad][h_in], boxes of 8 rows x 256
  const SlotRow *slots;
  float *zws;            // partial planes [ks][max_tokens][R_pad]; the result goes to plane kMaxZSplits
  int32_t *counters;     // arrivals per (group, eight rank rows), zero between launches
  uint32_t *status;
  int32_t x_index, n_ksteps, ks, R_pad, max_tokens;
};
struct DecShrinkBatch {
  CUtensorMap x[kDecInputs];  // [T][h_in], boxes of 1 row x 256
  DecShrinkSite site[kDecSites];
  int32_t n_sites, T, n_slots;
  const int32_t *ids;
  PlanView pv;           // published by the last CTA
  int32_t *zero;         // the base launch's arrival counters
  int32_t n_zero;
};

// The shape of the base launch for N columns and rank strides up to R_pad.
constexpr size_t kDecSmemBudget = 226 * 1024;
struct DecShape {
  int32_t stages, exp_stages, exp_bytes, n_acc, tmem_cols;
  size_t smem;
};
DecShape decode_sites_shape(int32_t N, int32_t R_pad);
cudaError_t decode_sites_set_smem_limit();
cudaError_t launch_decode_sites(const DecBatch &b, const DecShape &shape, int32_t grid, bool pdl, cudaStream_t stream);
cudaError_t launch_decode_sites_shrink(const DecShrinkBatch &b, int32_t grid, bool pdl, cudaStream_t stream);

}  // namespace edgelora
