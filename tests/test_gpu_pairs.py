"""The prefill kernels at the edges of their tiling: token tiles of 256 over a pair of CTAs, tiles taken off the launch
queue in long launches, runs of sites in one launch, the plan's two forms.  Against the CPU oracle, element by element.
"""
import numpy as np
import pytest

from paper_2507_01438_b200 import binding as B
from paper_2507_01438_b200 import workloads as wl
from helpers import assert_parity, oracle_of
from gpu_helpers import from_dev_bf16, make_pool, run_gpu, to_dev_bf16
from test_gpu_parity import check_plan, random_workload
from test_gpu_siteset import make_sites, mixed_ids, run_set

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,h_in,h_out,max_rank", [
    (257, 64, 8, 16),       # one token in the second token tile, one W chunk
    (384, 72, 264, 32),     # the follower's half of the last tile is empty
    (385, 520, 1000, 64),   # one token in it
    (513, 264, 40000, 16),  # more than four waves of tiles: the launch queue
    (1100, 1032, 2088, 64),
])
def test_tile_edges(T, h_in, h_out, max_rank):
    ranks = [max_rank, 1, 0, max_rank // 2, 8]
    w = random_workload(7 * T + h_out, T, h_in, h_out, ranks=ranks, max_rank=max_rank)
    rng = np.random.Generator(np.random.PCG64(T))
    n = 40   # decode tokens on every loaded adapter and on none, then runs that cross the tiles' borders
    cuts = np.sort(rng.choice(np.arange(n + 1, T), size=4, replace=False))
    lengths = np.diff(np.concatenate([[n], cuts, [T]]))
    w.ids = np.concatenate([rng.choice([-1, 0, 1, 3, 4], size=n), np.repeat([3, 0, -1, 4, 1], lengths)]).astype(np.int32)
    y, plan = run_gpu(w, return_plan=True)
    assert_parity(y, oracle_of(w), f"T={T} {h_in}->{h_out}")
    check_plan(plan, w.ids, w.n_slots)


@pytest.mark.parametrize("T,n_runs", [(2000, 1024), (2001, 1025), (4096, 4096), (4097, 3), (1025, 1)])
def test_plan_forms(T, n_runs):
    # the shared-memory form takes up to 4096 tokens in up to 1024 runs, the general form the others
    w = random_workload(T + n_runs, T, 64, 64, ranks=[8, 16, 4, 12, 16], max_rank=16)
    run = np.arange(T) * n_runs // T
    w.ids = ((run * 2) % 5 - (run % 7 == 3)).astype(np.int32)   # neighbours differ
    assert 1 + np.count_nonzero(np.diff(w.ids)) == n_runs
    y, plan = run_gpu(w, return_plan=True)
    assert_parity(y, oracle_of(w), f"{n_runs} runs")
    check_plan(plan, w.ids, w.n_slots)


def test_more_sites_and_inputs_than_one_launch_takes():
    ids = mixed_ids(5, 30, [(1, 200), (3, 90)], 4)
    shapes = [(64 + 8 * (i % 6), 72 + 8 * i) for i in range(35)]   # 35 sites on six inputs
    xs, sites = make_sites(11, len(ids), shapes, [16, 8, 4, 16], 16, ids)
    out = run_set(sites, xs, ids, 512)
    for w, y in zip(sites, out[0] if isinstance(out, tuple) else out):
        assert_parity(y, oracle_of(w), w.name)


def test_one_pool_at_two_sites_of_a_set():
    import torch
    ids = mixed_ids(6, 20, [(0, 300)], 3)
    _, (w1, w2) = make_sites(12, len(ids), [(128, 136), (128, 136)], [16, 8, 4], 16, ids)
    w2.adapters = w1.adapters          # tied adapters, another W and another input
    rng = np.random.Generator(np.random.PCG64(3))
    w2.x = wl.normal_bf16(rng, w1.x.shape, 1.0)
    pool = make_pool(w1)
    Ws = [to_dev_bf16(w.W) for w in (w1, w2)]
    s = B.edgelora_siteset_create([pool.handle, pool.handle], Ws, [0, 1], 2, len(ids))
    try:
        ys = [torch.empty((len(ids), 136), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        B.edgelora_siteset_run(s, [to_dev_bf16(w1.x), to_dev_bf16(w2.x)], torch.from_numpy(ids).cuda(), ys)
        assert pool.status() == (0, 0)
        for w, y in zip((w1, w2), ys):
            assert_parity(from_dev_bf16(y), oracle_of(w), w.name)
    finally:
        B.edgelora_siteset_destroy(s)
        pool.close()


@pytest.mark.parametrize("what", ["results", "input"])
def test_sites_of_a_set_that_share_memory(what):
    # two sites with one result buffer: the later one is seen; a result in an input's memory: the sites in order
    import torch
    ids = mixed_ids(8, 20, [(0, 300)], 3)
    T = len(ids)
    _, sites = make_sites(13, T, [(128, 128)] * 3, [16, 8, 4], 16, ids)
    pools = [make_pool(w) for w in sites]
    Ws = [to_dev_bf16(w.W) for w in sites]
    second = 1 if what == "input" else 0
    s = B.edgelora_siteset_create([p.handle for p in pools], Ws, [0, 0, second], 2, T)
    try:
        x = to_dev_bf16(sites[0].x)
        y = [torch.empty((T, 128), dtype=torch.bfloat16, device="cuda") for _ in range(3)]
        if what == "results":
            y[2] = y[0]
        B.edgelora_siteset_run(s, [x, y[0]], torch.from_numpy(ids).cuda(), y)
        if what == "input":
            sites[2].x = y[0].view(torch.int16).cpu().numpy().view(np.uint16)
        for i in ([1, 2] if what == "results" else [0, 1, 2]):
            assert_parity(from_dev_bf16(y[i]), oracle_of(sites[i]), sites[i].name)
        assert all(p.status() == (0, 0) for p in pools)
    finally:
        B.edgelora_siteset_destroy(s)
        for p in pools:
            p.close()


@pytest.mark.parametrize("T,n_runs", [
    (700, 511), (700, 512), (700, 513),    # runs ordered by counting, and by the sorting network
    (1030, 1030), (2049, 2047),            # more than one run per thread; the network's padding lies past the keys
    (4095, 4095), (4098, 4098),            # the last batch of the shared-memory form, the general form
])
def test_plan_orders(T, n_runs):
    w = random_workload(T + n_runs, T, 64, 64, ranks=[8, 16, 4, 0, 16, 2, 5], max_rank=16)
    rng = np.random.Generator(np.random.PCG64(n_runs))
    per_run = np.cumsum(rng.integers(1, 7, size=n_runs)) % 7     # neighbours differ
    w.ids = np.array([-1, 0, 1, 2, 4, 5, 6], np.int32)[per_run][np.arange(T) * n_runs // T]
    assert 1 + np.count_nonzero(np.diff(w.ids)) == n_runs
    y, plan = run_gpu(w, return_plan=True)
    assert_parity(y, oracle_of(w), f"T={T}")
    check_plan(plan, w.ids, w.n_slots)
