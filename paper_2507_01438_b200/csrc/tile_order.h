// The arithmetic of the pair kernel's walks that can be worked out without a GPU (plain C++, also compiled by the host
// compiler): the order of the tiles of a launch, the end of an operand ring.
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

}  // namespace edgelora
