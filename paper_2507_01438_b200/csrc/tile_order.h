// The arithmetic of the tile kernels' walks that can be worked out without a GPU (plain C++, also compiled by the host
// compiler): the order of the tiles of a launch, the end of an operand ring, the parts of the shrink's gather tiles.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define EDGELORA_HD __host__ __device__ __forceinline__
#else
#define EDGELORA_HD inline
#endif

namespace edgelora {

// The tile of a position of the launch's list: site, token tile, W tile.  Token tiles run fastest, so that
// neighbouring pairs share a W tile; the first token tile of a column moves with the column, because in a
// serving batch the first token tile holds the decode tokens (many adapters, many LoRA K blocks) and a
// fixed order would hand it to the same pairs again and again.
// `site` is the site of the role's tile before and becomes this tile's.  The positions of a role's tiles need not
// rise: the launch queue names the clusters that have not started in no promised order.
struct Tile {
  int32_t s, m, n;
};
template <typename Batch>
EDGELORA_HD Tile tile_at(const Batch &b, int32_t tile, int32_t &site) {
  while (site > 0 && tile < b.site[site - 1].tile_end) --site;
  while (tile >= b.site[site].tile_end) ++site;
  const int32_t local = tile - (site > 0 ? b.site[site - 1].tile_end : 0);
  Tile t;
  t.s = site;
  t.n = local / b.n_mtiles;
  t.m = (local + t.n) % b.n_mtiles;
  return t;
}

// Where in its ring a producer that has filled `used` stages in all begins to wait for the last use of each stage that
// it has filled: `stage` with parity `phase` ^ 1, then on around the ring, min(used, nstages) times.  A ring that was
// never filled once is waited for from its beginning (the stages behind the last one used were never filled, and a wait
// for them would pass at once).
struct RingPos {
  uint32_t stage, phase;
};
EDGELORA_HD RingPos ring_drain(uint32_t used, uint32_t nstages) {
  if (used < nstages) return RingPos{0u, 1u};
  return RingPos{used % nstages, (used / nstages) & 1u};
}

// Parts that the tokens of a gather tile of the shrink are cut into, each a tile of its own (a power of two, its logarithm
// here).  A tile goes through its tokens 64 at a time, one pass after the other over its K blocks: with hundreds of
// scattered tokens on a few adapters (and so a few tiles) the passes are what the launch takes.  As many parts as idle CTAs
// of the grid would take, and half as many again as an average tile has passes (tiles differ, and a part of two passes
// takes twice as long); tiles of one pass stay whole.  2048 tokens 4096 wide on 4 adapters: 344 -> 30 us, on 16 adapters
// 192 -> 36; 4096 tokens on 100 adapters by a power law 413 -> 160.
// n_tok tokens in n_tiles >= 1 tiles; items: what the launch has of them without parts (K splits, sites).
constexpr int32_t kGatherPass = 64;
EDGELORA_HD int32_t gather_parts_lg(int32_t n_tok, int32_t n_tiles, int32_t items, int32_t grid) {
  const int32_t passes = (n_tok + kGatherPass - 1) / kGatherPass;
  int32_t lp = 0;
  while ((1 << lp) < passes && (2 * (n_tiles << lp) < 3 * passes || (items << (lp + 1)) <= grid)) ++lp;
  return lp;
}
// The tokens [skip, skip + n) of a tile's n_tok that are in one of its parts: whole passes, except at the end.
struct GatherPart {
  int32_t skip, n;
};
EDGELORA_HD GatherPart gather_part(int32_t n_tok, int32_t part, int32_t lg_parts) {
  const int32_t passes = (n_tok + kGatherPass - 1) / kGatherPass;
  const int32_t n = ((passes + (1 << lg_parts) - 1) >> lg_parts) * kGatherPass;
  const int32_t skip = part * n < n_tok ? part * n : n_tok;
  return GatherPart{skip, n_tok - skip < n ? n_tok - skip : n};
}
// Gather tiles (in parts) of a site at most, for its arrival counters: batches up to max_tokens tokens in up to max_tiles
// tiles.  The last doubling leaves fewer than three times the passes, or no more items than the grid takes.
inline int64_t gather_tiles_max(int32_t max_tokens, int32_t max_tiles, int32_t grid) {
  const int64_t parts = 3 * (static_cast<int64_t>(max_tokens) / kGatherPass + 1);
  const int64_t most = parts > grid ? parts : grid;
  return most > max_tiles ? most : max_tiles;
}

}  // namespace edgelora
