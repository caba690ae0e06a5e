// What the kernel of decode_tile.cu is launched with: one linear site over a decode-sized batch.
#pragma once
#include "internal.cuh"

namespace edgelora {

constexpr int kTileMaxStages = 12;
constexpr int kTileMaxParts = 8;    // CTAs that share a tile: one cluster of portable size
constexpr size_t kTileSmemBudget = 226 * 1024;

struct DecTile {
  CUtensorMap w;         // W [h_out][h_in], boxes of 128 rows x 64
  CUtensorMap x;         // [T][h_in], boxes of N rows x 64
  CUtensorMap b;         // the pool's B blocks [S][h_out][R_pad], boxes of 128 rows x R_pad
  uint16_t *y;           // [T][h_out]
  const SlotRow *slots;
  const float *z;        // [max_tokens][R_pad], live groups of eight rank rows only
  uint32_t *status;
  const int32_t *ids;    // the caller's ids (validated again inside the kernel)
  int32_t T, h_out, kb, R_pad, n_slots;
  int32_t N;             // UMMA N: tokens rounded up to 16
  int32_t parts;         // CTAs of a cluster, which share a tile
  int32_t stages, exp_bytes, tmem_cols;
  long long wait_cycles;
};
struct DecTileShape {
  int32_t stages, exp_bytes, tmem_cols;
};
DecTileShape decode_tile_shape(int32_t N, int32_t R_pad);
// Whether the exchange of `parts` parts of T columns fits the rings' memory.
bool decode_tile_parts_fit(int32_t T, int32_t parts);
// Clusters of `parts` CTAs that the current device holds at once.
int32_t decode_tile_max_clusters(int32_t parts);
cudaError_t decode_tile_set_smem_limit();
cudaError_t launch_decode_tile(const DecTile &p, bool pdl, cudaStream_t stream);

}  // namespace edgelora
