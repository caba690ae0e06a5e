// The work of a decode launch as one list of units, cut into equal runs for its CTAs (plain C++, also compiled by the
// host compiler): the runs, and the pieces of tiles that a run goes through.
#pragma once
#include <stdint.h>

#include "tile_order.h"

namespace edgelora {

// n units over p runs: run i is [begin(i), begin(i + 1)), the first n % p of them one unit longer.
struct Runs {
  int32_t q, r;
  EDGELORA_HD Runs(int32_t n, int32_t p) : q(n / p), r(n - n / p * p) {}
  EDGELORA_HD int32_t begin(int32_t i) const { return i * q + (i < r ? i : r); }
  EDGELORA_HD int32_t of(int32_t unit) const {  // the run that holds a unit (there are units)
    const int32_t wide = r * (q + 1);
    return unit < wide ? unit / (q + 1) : r + (unit - wide) / q;
  }
};

// Expand units of a tile (one for 64 rank columns of B: as many bytes as a K block of W), of n stages.
EDGELORA_HD int32_t expand_units(int32_t n_stages, int32_t R_pad) { return (n_stages * R_pad + 63) >> 6; }
// Stages that T tokens on adapters of n_slots slots make at most, `tok` tokens of an adapter in a stage.
EDGELORA_HD int32_t expand_stages_max(int32_t T, int32_t n_slots, int32_t tok) {
  const int32_t g = T < n_slots ? T : n_slots;
  return g + (T - g) / tok;
}
// Runs of a launch of n units on a device of p SMs: four units each at least.
EDGELORA_HD int32_t run_count(int32_t n, int32_t p) {
  const int32_t most = n / 4 > 1 ? n / 4 : 1;
  return most < p ? most : p;
}

// What a run does of one tile: its expand stages' units first, the units of its K blocks behind them.
struct Piece {
  int32_t s, tile;   // site, W row tile of the site
  int32_t e0, e1;    // units of the expand
  int32_t kb0, kb1;  // K blocks
  int32_t first;     // the tile's first unit in the launch's list
  int32_t units;     // units of the tile
  EDGELORA_HD int32_t size() const { return (e1 - e0) + (kb1 - kb0); }
};
// The piece at unit `u` of a run that ends at `end`; `site` is the site of the piece before and becomes this one's.
// site_end[i]: units of the sites up to i; expand[i], kb[i]: expand units and K blocks of a tile of site i.
template <typename Expand, typename Kb>
EDGELORA_HD Piece piece_at(int32_t u, int32_t end, const int32_t *site_end, const Expand &expand, const Kb &kb,
                           int32_t &site) {
  while (u >= site_end[site]) ++site;
  Piece p;
  p.s = site;
  const int32_t base = site > 0 ? site_end[site - 1] : 0, ne = expand(site);
  p.units = ne + kb(site);
  p.tile = (u - base) / p.units;
  p.first = base + p.tile * p.units;
  const int32_t o0 = u - p.first, o1 = end - p.first < p.units ? end - p.first : p.units;
  p.e0 = o0 < ne ? o0 : ne;
  p.e1 = o1 < ne ? o1 : ne;
  p.kb0 = o0 > ne ? o0 - ne : 0;
  p.kb1 = o1 > ne ? o1 - ne : 0;
  return p;
}

}  // namespace edgelora
