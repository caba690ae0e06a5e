"""The order in which the pair kernel's roles walk a launch's tiles, the end of its operand ring, and the parts of the
shrink's gather tiles, on the CPU: csrc/tile_order.h is plain C++ and is
compiled here with the host compiler.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "tile_order.h"
struct Site { int32_t tile_end; };
struct Batch { Site site[32]; int32_t n_sites, n_mtiles; };
extern "C" void walk(int32_t n_sites, const int32_t *tile_end, int32_t n_mtiles, int32_t n, const int32_t *tiles, int32_t *out) {
  Batch b;
  b.n_sites = n_sites;
  b.n_mtiles = n_mtiles;
  for (int i = 0; i < n_sites; ++i) b.site[i].tile_end = tile_end[i];
  int32_t site = 0;
  for (int i = 0; i < n; ++i) {
    const edgelora::Tile t = edgelora::tile_at(b, tiles[i], site);
    out[3 * i] = t.s; out[3 * i + 1] = t.m; out[3 * i + 2] = t.n;
  }
}
extern "C" int32_t drain(uint32_t used, uint32_t nstages, uint32_t *stage, uint32_t *phase) {
  const edgelora::RingPos p = edgelora::ring_drain(used, nstages);
  *stage = p.stage;
  *phase = p.phase;
  return 0;
}
extern "C" int32_t parts_lg(int32_t n_tok, int32_t n_tiles, int32_t items, int32_t grid) {
  return edgelora::gather_parts_lg(n_tok, n_tiles, items, grid);
}
extern "C" void part(int32_t n_tok, int32_t p, int32_t lg, int32_t *out) {
  const edgelora::GatherPart g = edgelora::gather_part(n_tok, p, lg);
  out[0] = g.skip;
  out[1] = g.n;
}
extern "C" int64_t tiles_max(int32_t max_tokens, int32_t max_tiles, int32_t grid) {
  return edgelora::gather_tiles_max(max_tokens, max_tiles, grid);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("tile_order")
    src, out = d / "t.cpp", d / "t.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_2507_01438_b200", "csrc"), str(src), "-o", str(out)], check=True)
    return ctypes.CDLL(str(out))


@pytest.mark.parametrize("n_mtiles,w_tiles", [(1, [3]), (2, [16, 1, 4]), (9, [16, 4, 4, 16, 56, 56, 16]), (3, [1] * 32)])
@pytest.mark.parametrize("order", ["rising", "falling", "shuffled"])
def test_every_tile_is_found_in_any_order(lib, n_mtiles, w_tiles, order):
    # the launch queue promises no order of its answers
    ends = np.cumsum(np.array(w_tiles) * n_mtiles).astype(np.int32)
    tiles = np.arange(ends[-1], dtype=np.int32)
    if order == "falling":
        tiles = tiles[::-1].copy()
    elif order == "shuffled":
        np.random.default_rng(len(w_tiles)).shuffle(tiles)
    out = np.full((len(tiles), 3), -99, np.int32)
    ptr = lambda a: a.ctypes.data_as(ctypes.POINTER(ctypes.c_int32))
    lib.walk(len(ends), ptr(ends), n_mtiles, len(tiles), ptr(tiles), ptr(out))
    site = np.searchsorted(ends, tiles, side="right")
    local = tiles - np.concatenate([[0], ends[:-1]])[site]
    n = local // n_mtiles
    assert np.array_equal(out, np.stack([site, (local + n) % n_mtiles, n], axis=1))


@pytest.mark.parametrize("nstages", [1, 2, 6, 8])
def test_the_drain_waits_for_the_last_use_of_every_stage(lib, nstages):
    # a stage's barrier after k completed uses: a wait with parity p passes when the phase of parity p is over,
    # that is when (k - 1) % 2 == p, and on a barrier never used (k = 0) for parity 1
    for used in range(0, 4 * nstages + 1):
        stage, phase = ctypes.c_uint32(), ctypes.c_uint32()
        lib.drain(ctypes.c_uint32(used), ctypes.c_uint32(nstages), ctypes.byref(stage), ctypes.byref(phase))
        s, ph = stage.value, phase.value
        waited = []
        for _ in range(min(used, nstages)):
            uses = (used - s + nstages - 1) // nstages      # fills of this stage
            passes_after = lambda k: (k - 1) % 2 == (ph ^ 1)
            assert uses >= 1 and passes_after(uses) and not passes_after(uses - 1), (used, s, ph)
            waited.append(s)
            s += 1
            if s == nstages:
                s, ph = 0, ph ^ 1
        assert sorted(waited) == list(range(min(used, nstages)))


def test_the_parts_of_a_gather_tile_are_its_tokens_in_whole_passes(lib):
    out = (ctypes.c_int32 * 2)()
    for n_tok in (0, 1, 63, 64, 65, 300, 1024, 1025, 32768):
        for lg in range(0, 10):
            at = 0
            for p in range(1 << lg):
                lib.part(n_tok, p, lg, out)
                assert out[0] == at and out[1] >= 0
                assert out[1] % 64 == 0 or out[0] + out[1] == n_tok
                at += out[1]
            assert at == n_tok


def test_the_gather_tiles_of_a_batch_fit_the_arrival_counters(lib):
    lib.tiles_max.restype = ctypes.c_int64
    grid = 148
    for max_tokens in (257, 1000, 4096, 9500, 32768):
        for n_slots in (1, 3, 100, 65534):
            for r_pad in (16, 32, 64):
                max_tiles = -(-min(max_tokens, n_slots) * r_pad // 128)
                bound = lib.tiles_max(max_tokens, max_tiles, grid)
                for n_tok in sorted({1, 64, 65, 300, max_tokens // 3, max_tokens}):
                    for n_tiles in sorted({1, 2, 3, 7, max_tiles // 5, max_tiles}):
                        if not 1 <= n_tiles <= min(max_tiles, n_tok):
                            continue
                        for splits, n_sites in ((1, 1), (8, 1), (2, 32)):
                            lg = lib.parts_lg(n_tok, n_tiles, n_tiles * splits * n_sites, grid)
                            assert (n_tiles << lg) <= bound and (1 << lg) < 2 * max(1, -(-n_tok // 64))
                            assert lg == 0 or n_tok > 64
