// What the tensor-core shrink of shrink_tiles.cu is launched with: a run of linear sites over one batch.
#pragma once
#include "internal.cuh"

namespace edgelora {

constexpr int kTileSites = 32;   // sites of one launch at most
constexpr int kTileInputs = 4;   // distinct inputs of one launch at most
constexpr int kTileStages = 8;
constexpr int kTileGatherN = 64;  // token rows of one gather pass
constexpr size_t kTileTailBytes = 1024;

struct ShrinkSite {
  CUtensorMap a;           // the A blocks as one matrix [n_slots * R_pad][h_in], boxes of R_pad rows x 64
  const SlotRow *slots;
  float *zws;              // partial planes [splits][max_tokens][R_pad]; the result goes to plane kMaxZSplits
  int32_t *tile_counters;  // arrivals per tile, zero between launches
  uint32_t *status;
  int32_t x_index;         // which of the launch's inputs
  int32_t kb_total, R_pad, max_tokens;
  int32_t splits;          // K splits of a tile; 0: gather tiles only, split count chosen on the device
};
template <int kSites>
struct ShrinkBatch {
  static constexpr int kInputs = kSites == 1 ? 1 : kTileInputs;
  CUtensorMap x[kInputs];   // [T][h_in], boxes of 128 rows x 64
  CUtensorMap xg[kInputs];  // the same in boxes of one row, for the gather copies
  ShrinkSite site[kSites];
  int32_t n_sites, T, n_slots;
  int32_t z_bf16;           // 1: the result as bf16, zero at and past the rank; 0: as fp32
  const int32_t *sgmv_tiles, *counts, *perm_short, *gs_short, *group_adapter, *ids_valid;  // of the plan all sites share
  long long wait_cycles;
};

cudaError_t shrink_tiles_set_smem_limit();
template <int kSites>
cudaError_t launch_shrink_tiles(const ShrinkBatch<kSites> &b, int32_t grid, bool pdl, cudaStream_t stream);

}  // namespace edgelora
