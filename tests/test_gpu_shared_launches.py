"""Sets of sites whose launches are shared, in the forms that the ordinary set tests do not take: inputs of different
widths at one address, results that are inputs, waits that run out.  Against the CPU oracle, element by element.
"""
import numpy as np
import pytest

from paper_2507_01438_b200 import binding as B
from paper_2507_01438_b200 import workloads as wl
from helpers import assert_parity, oracle_of
from gpu_helpers import from_dev_bf16, make_pool, to_dev_bf16
from test_gpu_parity import random_workload
from test_gpu_siteset import make_sites, mixed_ids

pytestmark = pytest.mark.gpu


class SetOf:
    """Pools, weights and the set of some sites; ``inputs`` gives each site's input number."""

    def __init__(self, sites, inputs, max_tokens=0):
        import torch
        self.sites = sites
        T = sites[0].T
        self.pools = [make_pool(w, max_tokens or T) for w in sites]
        self.Ws = [to_dev_bf16(w.W) for w in sites]
        self.ids = torch.from_numpy(sites[0].ids).cuda()
        self.ys = [torch.full((T, w.h_out), float("nan"), dtype=torch.bfloat16, device="cuda") for w in sites]
        self.handle = B.edgelora_siteset_create([p.handle for p in self.pools], self.Ws, inputs, max(inputs) + 1,
                                                max_tokens or T)

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        B.edgelora_siteset_destroy(self.handle)
        for p in self.pools:
            p.close()

    def run(self, xs, stream=None):
        B.edgelora_siteset_run(self.handle, xs, self.ids, self.ys, stream)

    def check(self, what="", rows=None):
        for p in self.pools:
            assert p.status() == (0, 0)
        for w, y in zip(self.sites, self.ys):
            got = from_dev_bf16(y)
            assert_parity(got if rows is None else got[rows], oracle_of(w, rows), f"{what} {w.name}")


def test_inputs_of_different_widths_at_one_address():
    # input 0 is [T][128], input 1 the first T * 64 values of the same buffer as [T][64]
    ids = mixed_ids(21, 20, [(0, 300)], 3)
    T = len(ids)
    xs, sites = make_sites(22, T, [(128, 136), (64, 72), (128, 64), (64, 264)], [16, 8, 4], 16, ids)
    for w in sites:
        if w.h_in == 64:
            w.x = np.ascontiguousarray(xs[128].reshape(-1)[:T * 64].reshape(T, 64))
    with SetOf(sites, [0, 1, 0, 1]) as s:
        wide = to_dev_bf16(xs[128])
        s.run([wide, wide.view(-1)[:T * 64].view(T, 64)])
        s.check()


@pytest.mark.parametrize("options", [{}, {B.OPT_PDL: 2}, {B.OPT_PDL: 0}, {B.OPT_REGIME: 2}])
@pytest.mark.parametrize("T", [20, 200, 320])
def test_a_result_that_is_an_input_of_later_sites(T, options):
    import torch
    # site 0 streams a wide W and writes into input 1, which sites 1 and 3 read; site 2 does not
    ids = mixed_ids(23, 20, [(0, T - 20)], 3)
    xs, sites = make_sites(24, T, [(4096, 256), (256, 264), (4096, 136), (256, 72)], [16, 8, 4], 16, ids)
    with SetOf(sites, [0, 1, 0, 1]) as s:
        for p in s.pools:
            for option, value in options.items():
                B.edgelora_pool_set_option(p.handle, option, value)
        for _ in range(3):
            s.ys[0].fill_(float("nan"))   # a site that reads too early reads these
            s.run([to_dev_bf16(xs[4096]), s.ys[0]])
            sites[1].x = sites[3].x = s.ys[0].view(torch.int16).cpu().numpy().view(np.uint16)
            s.check(f"T={T}")


@pytest.mark.parametrize("how", ["chained set", "planned calls"])
@pytest.mark.parametrize("T", [24, 150])
def test_the_first_reader_of_a_plan_starts_behind_the_kernel_that_wrote_it(T, how):
    # Other ids in every step, steps issued while the GPU is busy, pools that allow overlap with earlier work: a kernel that
    # starts under the plan kernel reads the ids of the step before.  Same bits as with a wait behind every launch.
    import torch
    rng = np.random.Generator(np.random.PCG64(71))
    xs, sites = make_sites(72, T, [(1024, 256), (256, 264), (1024, 136)], [16, 8, 4, 16, 12], 16,
                           rng.integers(-1, 5, size=T).astype(np.int32))
    steps = [torch.from_numpy(rng.integers(-1, 5, size=T).astype(np.int32)).cuda() for _ in range(6)]
    with SetOf(sites, [0, 1, 0]) as s:
        plan = B.edgelora_plan_create(T, 5)
        for p in s.pools:
            B.edgelora_pool_set_option(p.handle, B.OPT_PDL, 2)
        x, busy = to_dev_bf16(xs[1024]), torch.randn(4096, 4096, device="cuda")

        def run(wait):
            sync = torch.cuda.synchronize if wait else (lambda: None)
            outs = [[torch.full_like(y, float("nan")) for y in s.ys] for _ in steps]
            torch.cuda.synchronize()
            for _ in range(4):
                torch.mm(busy, busy)
            for ids, ys in zip(steps, outs):
                if how == "chained set":
                    B.edgelora_siteset_run(s.handle, [x, ys[0]], ids, ys)
                else:
                    B.edgelora_plan_build(plan, ids)
                    for i in (0, 2):
                        sync()
                        B.edgelora_lora_linear_planned(s.pools[i].handle, plan, s.Ws[i], x, ys[i])
                sync()
            torch.cuda.synchronize()
            return [[y.view(torch.int16).cpu().numpy() for y in ys] for ys in outs]

        for got, want in zip(run(False), run(True)):
            for a, b in zip(got, want):
                assert np.array_equal(a, b)
        assert [p.status() for p in s.pools] == [(0, 0)] * 3
        B.edgelora_plan_destroy(plan)


def shorten_waits(pool, on=True):
    # 1024 cycles, and what a single try of a barrier may take: far less than the longest waits of these calls.  The
    # kernels give up, wait for what they have in flight, report and return; sync_status brings the pool back
    B.edgelora_pool_set_option(pool.handle, B.OPT_WAIT_CYCLES, 1 if on else 0)


@pytest.mark.parametrize("T,h_in,h_out,options", [
    (300, 2048, 264, {}),                        # shrink and pair kernel, tiles dealt out
    (513, 1032, 40000, {}),                      # tiles off the launch queue
    (40, 2048, 264, {B.OPT_REGIME: 2}),          # gather tiles only
    (24, 4096, 512, {}),                         # decode in one launch
    (200, 14336, 520, {}),                       # decode, shrink and tile kernel
])
def test_a_call_whose_waits_run_out_reports_and_leaves_the_pool_usable(T, h_in, h_out, options):
    import torch
    w = random_workload(31, T, h_in, h_out, ranks=[16, 8, 4], max_rank=16)
    rows = np.unique(np.linspace(0, T - 1, 24).astype(int))
    pool = make_pool(w)
    try:
        for option, value in options.items():
            B.edgelora_pool_set_option(pool.handle, option, value)
        W, x, ids = to_dev_bf16(w.W), to_dev_bf16(w.x), torch.from_numpy(w.ids).cuda()
        for _ in range(2):
            shorten_waits(pool)
            pool.linear(W, x, ids)
            assert pool.status() == (B.ERR_TIMEOUT, B.STATUS_TIMEOUT)
            shorten_waits(pool, False)
            y = pool.linear(W, x, ids)
            assert pool.status() == (0, 0)
            assert_parity(from_dev_bf16(y)[rows], oracle_of(w, rows), "after the time-out")
    finally:
        pool.close()


def test_a_wait_that_runs_out_in_a_shared_launch_is_reported_by_every_site():
    # more items and tiles than the first round of CTAs takes, in a launch that deals its tiles out: those of the last
    # site (two K parts per shrink tile) need not be reached.  Its pool reports all the same, and its arrival counters are
    # back in place for the next run
    T = 513
    ids = mixed_ids(33, 30, [(i % 3, 40) for i in range(11)] + [(0, 43)], 3)
    shapes = [(2048, 8192)] + [(256, 72)] * 18 + [(4096, 64)]
    _, sites = make_sites(34, T, shapes, [16, 8, 4], 16, ids)
    xs = {w.h_in: to_dev_bf16(w.x) for w in sites}
    with SetOf(sites, [0] + [1] * 18 + [2]) as s:
        for _ in range(2):
            for p in s.pools:
                shorten_waits(p)
            s.run([xs[2048], xs[256], xs[4096]])
            assert [p.status() for p in s.pools] == [(B.ERR_TIMEOUT, B.STATUS_TIMEOUT)] * len(sites)
            for p in s.pools:
                shorten_waits(p, False)
            for _ in range(2):
                s.run([xs[2048], xs[256], xs[4096]])
                s.check("after the time-out", np.array([0, 17, 29, 30, 111, 512]))


@pytest.mark.parametrize("sites", [1, 3])
def test_a_long_run_on_an_empty_slot_raises_the_status(sites):
    # 300 tokens of one prompt on a slot with nothing loaded: base-only, and the pool says so
    ids = mixed_ids(41, 10, [(0, 60), (1, 300), (2, 40)], 3)
    ids[:10] = 0
    _, ws = make_sites(42, len(ids), [(256, 136), (256, 72), (4096, 64)][:sites], [16, 0, 8], 16, ids)
    xs = [to_dev_bf16(ws[i].x) for i in ([0] if sites == 1 else [0, 2])]
    with SetOf(ws, [0, 0, 1][:sites]) as s:
        s.run(xs)
        assert [p.status() for p in s.pools] == [(B.ERR_SLOT_EMPTY, B.STATUS_SLOT_EMPTY)] * sites
        for w in ws:
            w.ids = np.where(ids == 1, -1, ids).astype(np.int32)
        s.check()


def test_pools_with_their_own_wait_limits_do_not_share_a_launch():
    ids = mixed_ids(43, 20, [(0, 300)], 3)
    _, ws = make_sites(44, len(ids), [(128, 72)] * 4, [16, 8, 4], 16, ids)
    with SetOf(ws, [0] * 4) as s:
        B.edgelora_pool_set_option(s.pools[2].handle, B.OPT_WAIT_CYCLES, 1 << 20)
        s.run([to_dev_bf16(ws[0].x)])
        s.check()
        assert [B.edgelora_pool_last_launch(p.handle)["launches"] for p in s.pools] == [2, 0, 2, 2]


def test_an_input_still_on_its_way_ends_a_run_in_front_of_its_first_reader():
    import torch
    ids = mixed_ids(45, 20, [(0, 300)], 3)
    xs, ws = make_sites(46, len(ids), [(256, 72), (256, 64), (128, 72), (256, 136)], [16, 8, 4], 16, ids)
    pin = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a).view(dt)).pin_memory()
    with SetOf(ws, [0, 0, 1, 0]) as s:
        ys = [None] * 3 + [torch.zeros((len(ids), 136), dtype=torch.int16).pin_memory()]
        B.edgelora_siteset_run_host(s.handle, [pin(xs[256], np.int16), pin(xs[128], np.int16)], pin(ids, np.int32), ys)
        assert [B.edgelora_pool_last_launch(p.handle)["launches"] for p in s.pools] == [2, 0, 2, 0]
        assert_parity(wl.bf16_bits_to_f32(ys[3].numpy().view(np.uint16)), oracle_of(ws[3]), ws[3].name)


@pytest.mark.parametrize("rank", [16, 32, 64])
@pytest.mark.parametrize("T,n_adapters", [(300, 3), (513, 40), (700, 300)])
def test_a_non_finite_adapter_reaches_its_own_tokens_only(T, n_adapters, rank):
    import torch
    # every third adapter has an infinity or NaN in its B; the others share token tiles with it
    rng = np.random.Generator(np.random.PCG64(T + rank))
    w = random_workload(T, T, 264, 392, ranks=[rank] * n_adapters, max_rank=rank)
    w.ids = rng.permutation(np.arange(T) % (n_adapters + 1) - 1).astype(np.int32)
    w.ids[60:100] = 1                                     # and a run of its own, in the first tile
    bad = np.isin(w.ids, np.arange(0, n_adapters, 3))
    want = oracle_of(w)
    for a in range(0, n_adapters, 3):
        w.adapters[a].B[:, a % rank] = 0x7F80 if a % 2 else 0x7FC0   # bfloat16 infinity, NaN
    pool = make_pool(w)
    try:
        got = from_dev_bf16(pool.linear(to_dev_bf16(w.W), to_dev_bf16(w.x), torch.from_numpy(w.ids).cuda()))
        assert pool.status() == (0, 0)
        assert_parity(got[~bad], want[~bad], "tokens on finite adapters and on none")
        assert not np.isfinite(got[bad]).any()
    finally:
        pool.close()


@pytest.mark.parametrize("T,h_out", [(300, 264), (513, 40000)])
def test_the_reported_grid_is_the_launch(T, h_out):
    # a tile per pair while the pairs of the device hold them, a cluster per tile off the launch queue
    import torch
    w = random_workload(51, T, 64, h_out, ranks=[16], max_rank=16)
    pool = make_pool(w)
    try:
        pool.linear(to_dev_bf16(w.W), to_dev_bf16(w.x), torch.from_numpy(w.ids).cuda())
        info = B.edgelora_pool_last_launch(pool.handle)
        tiles = -(-T // 256) * -(-h_out // info["n_tile"])
        assert info["gemm_grid"] == 2 * tiles
    finally:
        pool.close()


def test_sites_of_different_rank_strides_off_the_launch_queue():
    T = 513
    ids = mixed_ids(61, 40, [(0, 200), (2, 31), (1, 242)], 4)
    sites = []
    for i, (h_in, h_out, rank) in enumerate([(264, 16384, 16), (72, 16384, 64), (1032, 2056, 32), (264, 136, 64)]):
        sites += make_sites(62 + i, T, [(h_in, h_out)], [rank, rank // 2, 4, rank], rank, ids)[1]
    with SetOf(sites, [0, 1, 2, 3]) as s:
        s.run([to_dev_bf16(w.x) for w in sites])
        info = B.edgelora_pool_last_launch(s.pools[0].handle)
        assert info["launches"] == 2 and info["gemm_grid"] > 148     # one run, a cluster per tile
        s.check(rows=np.array([0, 7, 39, 40, 239, 240, 255, 256, 270, 271, 400, 512]))


def test_more_sites_than_one_launch_takes_on_few_inputs():
    ids = mixed_ids(65, 20, [(1, 250), (0, 40)], 3)
    shapes = [((64, 128, 72)[i % 3], 64 + 8 * i) for i in range(35)]   # 35 sites on three inputs: 32 and 3
    xs, sites = make_sites(66, len(ids), shapes, [16, 8, 4], 16, ids)
    with SetOf(sites, [i % 3 for i in range(35)]) as s:
        s.run([to_dev_bf16(xs[h]) for h in (64, 128, 72)])
        s.check()
        assert [B.edgelora_pool_last_launch(p.handle)["launches"] for p in s.pools] == [2] + [0] * 31 + [2, 0, 0]


def test_a_captured_set_of_a_large_batch():
    import torch
    ids = mixed_ids(67, 30, [(1, 250), (0, 60)], 3)
    xs, sites = make_sites(68, len(ids), [(256, 264), (512, 128), (256, 520)], [16, 8, 4], 16, ids)
    rng = np.random.Generator(np.random.PCG64(69))
    with SetOf(sites, [0, 1, 0]) as s:
        x = [to_dev_bf16(xs[256]), to_dev_bf16(xs[512])]
        for p in s.pools:
            B.edgelora_pool_wait_loads(p.handle)
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        s.run(x, stream)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            s.run(x, stream)
        for _ in range(2):                 # the replay reads what the buffers hold now
            for i, h in ((0, 256), (1, 512)):
                new = wl.normal_bf16(rng, xs[h].shape, 1.0)
                x[i].copy_(to_dev_bf16(new))
                for w in sites:
                    if w.h_in == h:
                        w.x = new
            for y in s.ys:
                y.fill_(float("nan"))
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                graph.replay()
            stream.synchronize()
            s.check("replay")
