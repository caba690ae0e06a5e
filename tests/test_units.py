"""The cut of a decode launch's work into runs, on the CPU: csrc/units.h is plain C++ and is compiled here with the host
compiler.  Every unit of every tile is done once, and the runs that share a tile are the ones the kernel takes for them.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "units.h"
extern "C" int32_t pieces(int32_t n_sites, const int32_t *tiles, const int32_t *expand, const int32_t *kb, int32_t p,
                          int32_t *out) {
  int32_t site_end[32], n = 0;
  for (int i = 0; i < n_sites; ++i) site_end[i] = n += tiles[i] * (expand[i] + kb[i]);
  const edgelora::Runs runs(n, p);
  const auto e = [&](int32_t s) { return expand[s]; };
  const auto k = [&](int32_t s) { return kb[s]; };
  int32_t count = 0;
  for (int32_t r = 0; r < p; ++r) {
    int32_t site = 0;
    for (int32_t u = runs.begin(r); u < runs.begin(r + 1);) {
      const edgelora::Piece x = edgelora::piece_at(u, runs.begin(r + 1), site_end, e, k, site);
      u += (x.e1 - x.e0) + (x.kb1 - x.kb0);
      const int32_t row[] = {r, x.s, x.tile, x.e0, x.e1, x.kb0, x.kb1, x.first, x.units,
                             runs.of(x.first), runs.of(x.first + x.units - 1)};
      for (int j = 0; j < 11; ++j) out[11 * count + j] = row[j];
      ++count;
    }
  }
  return count;
}
"""


SOURCE += r"""
extern "C" int32_t stages_max(int32_t T, int32_t n_slots, int32_t tok) { return edgelora::expand_stages_max(T, n_slots, tok); }
extern "C" int32_t run_count(int32_t n, int32_t p) { return edgelora::run_count(n, p); }
"""


@pytest.fixture(scope="module")
def units(tmp_path_factory):
    d = tmp_path_factory.mktemp("units")
    src, so = d / "u.cpp", d / "u.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-std=c++17", "-I",
                    os.path.join(ROOT, "paper_2507_01438_b200", "csrc"), "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("tiles,expand,kb,runs", [
    ([1], [0], [1], 1), ([1], [0], [4], 1), ([1], [3], [4], 7), ([40], [14], [49], 148), ([32], [109], [224], 148),
    ([32, 8, 8, 32, 112, 112, 32] * 4, [9] * 28, [64, 64, 64, 64, 64, 64, 224] * 4, 148),
    ([3, 1, 5], [0, 2, 1], [1, 1, 2], 9), ([1] * 32, [1] * 32, [1] * 32, 16), ([7], [0], [13], 22),
])
def test_every_unit_of_every_tile_is_done_once(units, tiles, expand, kb, runs):
    as_c = lambda v: np.ascontiguousarray(v, np.int32).ctypes.data_as(ctypes.c_void_p)
    out = np.zeros((sum(tiles) + 2 * runs + 64, 11), np.int32)
    n = units.pieces(len(tiles), as_c(tiles), as_c(expand), as_c(kb), runs, out.ctypes.data_as(ctypes.c_void_p))
    seen, by_tile = {}, {}
    for r, s, t, e0, e1, k0, k1, first, n_units, r0, r1 in out[:n].tolist():
        assert 0 <= t < tiles[s] and n_units == expand[s] + kb[s] and e1 + k1 > e0 + k0
        for unit in [("e", i) for i in range(e0, e1)] + [("k", i) for i in range(k0, k1)]:
            assert (s, t, unit) not in seen
            seen[s, t, unit] = r
        by_tile.setdefault((s, t, r0, r1), []).append(r)
    assert len(seen) == sum(a * (b + c) for a, b, c in zip(tiles, expand, kb))
    assert len(by_tile) == sum(tiles)
    starts = [r0 for _, _, r0, r1 in by_tile if r1 > r0]
    assert len(starts) == len(set(starts))           # a run begins one shared tile at most
    for (_, _, r0, r1), who in by_tile.items():
        assert who == list(range(r0, r1 + 1))        # the runs that add up a tile, a piece each


@pytest.mark.parametrize("T,n_slots", [(1, 1), (8, 1), (9, 1), (27, 64), (256, 3), (256, 40), (256, 1000)])
def test_a_workspace_for_the_most_stages_holds_every_batch(units, T, n_slots):
    # as many stages as the bound says are reached, none more; and a grid of the runs of the largest batch cuts a smaller one
    # as a grid of the whole device would
    rng = np.random.Generator(np.random.PCG64(T + n_slots))
    most = units.stages_max(T, n_slots, 8)
    worst = 0
    for k in range(60):
        few = rng.integers(1, n_slots + 1)
        n = np.bincount(rng.integers(0, few, size=rng.integers(1, T + 1)) if k else np.arange(T) % n_slots)
        worst = max(worst, int((-(-n // 8)).sum()))
        assert worst <= most
    groups = np.ones(min(T, n_slots), int)           # one token each, the others by whole stages on the first
    groups[0] += T - len(groups)
    assert int((-(-groups // 8)).sum()) == most or (T - len(groups)) % 8
    for n_max in (1, 7, 40, 590, 592, 10000):
        for n in {1, n_max // 3 + 1, n_max - 1 or 1, n_max}:
            assert units.run_count(n, units.run_count(n_max, 148)) == units.run_count(n, 148)
