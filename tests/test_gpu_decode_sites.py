"""Decode-sized batches through a set of sites: one shrink launch and one base launch for the whole set.  Against the CPU
oracle, element by element, at the edges of what the launches are cut into: batch sizes around the columns of the tensor
core and the tokens of an expand stage, widths that fill no K block, no K step and no row tile, tiles that several CTAs share.
"""
import numpy as np
import pytest

from paper_2507_01438_b200 import binding as B
from helpers import assert_parity, oracle_of
from gpu_helpers import from_dev_bf16, make_pool, to_dev_bf16
from test_gpu_shared_launches import SetOf
from test_gpu_siteset import check_plan, make_sites

pytestmark = pytest.mark.gpu

SHAPES = [(264, 136), (1032, 8), (264, 5000), (4096, 264), (1032, 392)]


def run_and_check(ids, ranks, max_rank, shapes=SHAPES, seed=5, again=1):
    xs, sites = make_sites(seed, len(ids), shapes, ranks, max_rank, ids)
    widths = sorted(xs)
    with SetOf(sites, [widths.index(w.h_in) for w in sites]) as s:
        for _ in range(again):
            for y in s.ys:
                y.fill_(float("nan"))
            s.run([to_dev_bf16(xs[h]) for h in widths])
            s.check(f"T={len(ids)}")
        check_plan(B.edgelora_plan_export(B.edgelora_siteset_plan(s.handle), len(ids)), ids, len(ranks))
        assert [B.edgelora_pool_last_launch(p.handle)["launches"] for p in s.pools] == [2] + [0] * (len(sites) - 1)


@pytest.mark.parametrize("T", [1, 7, 16, 17, 32, 33, 64, 65, 128, 129, 256])
def test_batch_sizes(T):
    rng = np.random.Generator(np.random.PCG64(T))
    ranks = [16, 8, 32, 4, 12, 32, 1]
    run_and_check(rng.integers(-1, len(ranks), size=T).astype(np.int32), ranks, 32, again=2)


@pytest.mark.parametrize("max_rank", [16, 32, 64])
@pytest.mark.parametrize("ids", ["one", "distinct", "base", "eights"])
def test_how_tokens_share_adapters(ids, max_rank):
    # all tokens on one adapter (many stages of one), each on its own, none on any, and groups of 8 and 9 tokens
    T = 72
    ids = {"one": np.full(T, 3), "distinct": np.random.Generator(np.random.PCG64(1)).permutation(T),
           "base": np.full(T, -1), "eights": np.repeat([5, -1, 2, 7, 0, 9, 4, 1, 8], [8, 9, 8, 9, 1, 16, 17, 2, 2])}[ids]
    ranks = [(max_rank, max_rank // 2, max(max_rank // 4, 4), max_rank - 3)[a % 4] for a in range(T)]
    run_and_check(ids.astype(np.int32), ranks, max_rank)


def test_tiles_of_many_runs_and_runs_of_many_tiles():
    # a wide input on few rows (every tile is shared by many CTAs) beside a narrow one on many
    ids = np.random.Generator(np.random.PCG64(2)).integers(-1, 6, size=40).astype(np.int32)
    run_and_check(ids, [16, 16, 8, 16, 4, 16], 16, [(14336, 128), (64, 20000), (14336, 8)])


@pytest.mark.parametrize("T", [20, 150])
def test_an_empty_slot_and_an_id_out_of_range(T):
    ids = np.random.Generator(np.random.PCG64(3)).integers(-1, 4, size=T).astype(np.int32)
    ids[[2, 5, 11]] = [1, 1, 4]
    _, sites = make_sites(6, T, [(264, 136), (264, 392)], [16, 0, 8, 16], 16, np.where(ids == 4, -1, ids))
    for w in sites:
        w.ids = ids
    import torch
    with SetOf(sites, [0, 0]) as s:
        s.run([to_dev_bf16(sites[0].x)])
        assert [p.status() for p in s.pools] == [(B.ERR_SLOT_EMPTY, B.STATUS_SLOT_EMPTY)] * 2
        rc, bits = B.edgelora_plan_sync_status(B.edgelora_siteset_plan(s.handle))
        assert (rc, bits) == (B.ERR_BAD_ADAPTER_ID, B.STATUS_BAD_ADAPTER_ID)
        for w in sites:
            w.ids = np.where((ids == 1) | (ids == 4), -1, ids).astype(np.int32)
        s.check()


def test_a_non_finite_adapter_reaches_its_own_tokens_only():
    ids = (np.arange(50) % 11 - 1).astype(np.int32)
    xs, sites = make_sites(7, 50, [(264, 136), (264, 392)], [16] * 10, 16, ids)
    want = [oracle_of(w) for w in sites]
    bad = np.isin(ids, [2, 7])
    for w in sites:
        w.adapters[2].B[:, 3], w.adapters[7].B[:, 15] = 0x7F80, 0x7FC0      # infinity, NaN
    with SetOf(sites, [0, 0]) as s:
        s.run([to_dev_bf16(xs[264])])
        for y, ref, w in zip(s.ys, want, sites):
            got = from_dev_bf16(y)
            assert_parity(got[~bad], ref[~bad], "tokens on finite adapters and on none")
            assert not np.isfinite(got[bad]).any()


def test_waits_that_run_out_are_reported_and_leave_the_set_usable():
    ids = np.random.Generator(np.random.PCG64(4)).integers(-1, 3, size=30).astype(np.int32)
    xs, sites = make_sites(8, 30, [(4096, 1000), (4096, 264)], [16, 8, 4], 16, ids)
    with SetOf(sites, [0, 0]) as s:
        x = to_dev_bf16(xs[4096])
        for _ in range(2):
            for p in s.pools:
                B.edgelora_pool_set_option(p.handle, B.OPT_WAIT_CYCLES, 1)
            s.run([x])
            assert [p.status() for p in s.pools] == [(B.ERR_TIMEOUT, B.STATUS_TIMEOUT)] * 2
            for p in s.pools:
                B.edgelora_pool_set_option(p.handle, B.OPT_WAIT_CYCLES, 0)
            s.run([x])
            s.check("after the time-out")


def test_sites_that_share_a_pool_or_a_result_keep_their_order():
    import torch
    ids = np.random.Generator(np.random.PCG64(9)).integers(-1, 3, size=24).astype(np.int32)
    xs, sites = make_sites(10, 24, [(264, 136), (264, 136), (264, 392)], [16, 8, 4], 16, ids)
    with SetOf(sites, [0, 0, 0]) as s:
        s.ys[1] = s.ys[0]                                 # the later site is to be seen
        s.run([to_dev_bf16(xs[264])])
        assert [B.edgelora_pool_last_launch(p.handle)["launches"] for p in s.pools] == [2, 2, 0]
        for i in (1, 2):
            assert_parity(from_dev_bf16(s.ys[i]), oracle_of(sites[i]), sites[i].name)
    pool = make_pool(sites[0], 24)
    W = to_dev_bf16(sites[0].W)
    h = B.edgelora_siteset_create([pool.handle, pool.handle], [W, W], [0, 0], 1, 24)
    try:
        ys = [torch.zeros(24, 136, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        B.edgelora_siteset_run(h, [to_dev_bf16(xs[264])], torch.from_numpy(ids).cuda(), ys)
        for y in ys:
            assert_parity(from_dev_bf16(y), oracle_of(sites[0]), "twice in a set")
        assert pool.status() == (0, 0)
    finally:
        B.edgelora_siteset_destroy(h)
        pool.close()


@pytest.mark.parametrize("options", [[2, 1], [2, 2], [1, 2]])
def test_a_run_starts_behind_the_work_in_front_of_the_set(options):
    # The input of every run but the first is a result of the run before it, and the GPU is still busy when the runs are
    # issued: a run that starts early reads what the buffers held before.  Same bits as with a wait behind every run.
    import torch
    ids = np.random.Generator(np.random.PCG64(12)).integers(-1, 3, size=40).astype(np.int32)
    xs, sites = make_sites(13, 40, [(1024, 1024), (1024, 392)], [16, 8, 4], 16, ids)
    with SetOf(sites, [0, 0]) as s:
        for p, value in zip(s.pools, options):
            B.edgelora_pool_set_option(p.handle, B.OPT_PDL, value)
        first, busy = to_dev_bf16(xs[1024]), torch.randn(4096, 4096, device="cuda")

        def chain(wait):
            outs = [[torch.full_like(y, float("nan")) for y in s.ys] for _ in range(6)]
            torch.cuda.synchronize()
            for _ in range(4):
                torch.mm(busy, busy)
            x = first
            for ys in outs:
                B.edgelora_siteset_run(s.handle, [x], s.ids, ys)
                x = ys[0]
                if wait:
                    torch.cuda.synchronize()
            torch.cuda.synchronize()
            return [[from_dev_bf16(y) for y in ys] for ys in outs]

        for got, want in zip(chain(False), chain(True)):
            for a, b in zip(got, want):
                assert np.array_equal(a, b) and np.isfinite(b).all()
        assert [p.status() for p in s.pools] == [(0, 0)] * 2


@pytest.mark.parametrize("pdl", [1, 2])
@pytest.mark.parametrize("T", [12, 130])
def test_several_runs_of_a_step_and_steps_in_a_row(T, pdl):
    # a pool that comes twice cuts a step into two runs, which use one workspace and one z in turn; nothing waits in between
    import torch
    ids = np.random.Generator(np.random.PCG64(14)).integers(-1, 4, size=T).astype(np.int32)
    xs, sites = make_sites(15, T, [(1032, 520), (1032, 136), (1032, 264)], [16, 8, 4, 16], 16, ids)
    pools, Ws, x = [make_pool(w, T) for w in sites], [to_dev_bf16(w.W) for w in sites], to_dev_bf16(xs[1032])
    order = [0, 1, 0, 2, 1]
    s = B.edgelora_siteset_create([pools[i].handle for i in order], [Ws[i] for i in order], [0] * 5, 1, T)
    try:
        for p in pools:
            B.edgelora_pool_set_option(p.handle, B.OPT_PDL, pdl)
        idt = torch.from_numpy(ids).cuda()
        steps = [[torch.full((T, sites[i].h_out), float("nan"), dtype=torch.bfloat16, device="cuda") for i in order]
                 for _ in range(4)]
        torch.cuda.synchronize()
        for ys in steps:
            B.edgelora_siteset_run(s, [x], idt, ys)
        for k, i in enumerate(order):
            got = [from_dev_bf16(ys[k]) for ys in steps]
            assert_parity(got[0], oracle_of(sites[i]), sites[i].name)
            assert all(np.array_equal(got[0], g) for g in got[1:])
        assert [p.status() for p in pools] == [(0, 0)] * 3
    finally:
        B.edgelora_siteset_destroy(s)
        for p in pools:
            p.close()
