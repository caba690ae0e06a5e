// What the pair kernel of prefill.cu is launched with: a run of linear sites over one batch.
#pragma once
#include <algorithm>

#include "internal.cuh"

namespace edgelora {

constexpr int kPairMaxStages = 8;
constexpr int kPairSites = 32;   // sites of one launch at most
constexpr int kPairInputs = 4;   // distinct inputs of one launch at most
constexpr int kYStageBytes = 4 * 32 * 128;  // epilogue: per warp 32 tokens x 64 bf16
constexpr size_t kPairTailBytes = 4096;
constexpr size_t kPairSmemBudget = 226 * 1024;

struct PairSite {
  CUtensorMap w;         // W [h_out][h_in], boxes of BN / 2 rows x 64
  CUtensorMap b;         // the pool's B blocks [S][h_out][R_pad], boxes of BN / 2 rows x R_pad
  uint16_t *y;           // [T][h_out]
  const SlotRow *slots;
  const uint4 *zb;       // z as bf16 [max_tokens][R_pad], zero at and past the true rank
  uint32_t *status;
  int32_t tile_end;      // tiles of this site and of those before it
  int32_t x_index;       // which of the launch's inputs
  int32_t h_out, kb_total, R_pad;
};
template <int kSites>
struct PairBatch {
  CUtensorMap x[kSites == 1 ? 1 : kPairInputs];  // [T][h_in], boxes of 128 rows x 64
  PairSite site[kSites];
  int32_t n_sites, T, n_slots;
  int32_t BN;        // W rows of a tile, a multiple of 32 up to 256
  int32_t stages, n_mtiles;
  const int32_t *ids_valid, *mt_count, *mt_list;  // of the plan all sites share
  long long wait_cycles;
};

int pair_stages(int BN);
// Launches of more than four tiles per pair take them off the launch queue (a cluster per tile); the others deal them to
// the pairs that fit the device (see launch_pair_gemm).
inline bool pair_queued(int32_t tiles, int32_t sms) { return tiles > 4 * std::max(1, sms / 2); }
inline int32_t pair_grid(int32_t tiles, int32_t sms) {  // CTAs
  return 2 * (pair_queued(tiles, sms) ? tiles : std::min(tiles, std::max(1, sms / 2)));
}
cudaError_t pair_set_smem_limit();
template <int kSites>
cudaError_t launch_pair_gemm(const PairBatch<kSites> &b, int32_t sms, bool pdl, cudaStream_t stream);

}  // namespace edgelora
