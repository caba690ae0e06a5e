"""Decode-sized batches of one site that take a shrink launch and a tile launch: more than 64 tokens, or too many for the row
tiles of the site.  Against the CPU oracle, element by element, at the edges: columns of the tensor core, token quads that
the parts of a tile finish, expand stages of one to eight tokens, rings that go round more than once.
"""
import numpy as np
import pytest

from paper_2507_01438_b200 import binding as B
from helpers import assert_parity, oracle_of
from gpu_helpers import from_dev_bf16, make_pool, run_gpu, to_dev_bf16
from test_gpu_parity import check_plan, random_workload

pytestmark = pytest.mark.gpu


def workload(seed, T, h_in, h_out, max_rank, n_adapters, ids=None):
    ranks = [(max_rank, max_rank // 2, max_rank - 3, max(max_rank // 4, 1))[a % 4] for a in range(n_adapters)]
    w = random_workload(seed, T, h_in, h_out, ranks=ranks, max_rank=max_rank)
    rng = np.random.Generator(np.random.PCG64(seed))
    w.ids = (rng.integers(-1, n_adapters, size=T) if ids is None else ids).astype(np.int32)
    return w


def run_and_check(w, splits=0):
    pool = make_pool(w)
    try:
        first = None
        for _ in range(2):
            y, plan = run_gpu(w, 1, pool=pool, return_plan=True, options={B.OPT_DECODE_SPLITS: splits})
            assert_parity(y, oracle_of(w), w.name)
            check_plan(plan, w.ids, w.n_slots)
            assert first is None or np.array_equal(first, y)
            first = y
        assert B.edgelora_pool_last_launch(pool.handle)["launches"] == 2
        return B.edgelora_pool_last_launch(pool.handle)["split_k"]
    finally:
        pool.close()


@pytest.mark.parametrize("max_rank", [16, 32, 64])
@pytest.mark.parametrize("T", [65, 80, 81, 127, 200, 256])
def test_batch_sizes_and_rank_strides(T, max_rank):
    run_and_check(workload(T, T, 1032, 392, max_rank, 70))


@pytest.mark.parametrize("splits", [1, 2, 3, 5, 7, 8])
@pytest.mark.parametrize("T", [67, 253])
def test_counts_of_parts(T, splits):
    # owners of unequal numbers of quads, or of none, K blocks that do not divide; a count whose exchange does not fit the
    # rings' memory is brought down
    got = run_and_check(workload(100 + T, T, 1288, 264, 64, 40), splits)
    assert got == splits if T == 67 else 1 <= got <= splits


@pytest.mark.parametrize("ids", ["one", "distinct", "base", "eights"])
def test_how_tokens_share_adapters(ids):
    T = 144
    v = {"one": np.full(T, 3), "distinct": np.random.Generator(np.random.PCG64(1)).permutation(T), "base": np.full(T, -1),
         "eights": np.repeat([5, -1, 2, 7, 0, 9, 4, 1, 8], [8, 9, 8, 9, 1, 16, 17, 2, 74])}[ids]
    run_and_check(workload(3, T, 520, 136, 32, T, v))


def test_few_tokens_on_many_row_tiles():
    run_and_check(workload(4, 20, 264, 10000, 16, 7))            # a row tile per CTA
    run_and_check(workload(5, 40, 512, 5128, 32, 50))            # too many tokens per owner for the one-launch path


def test_a_non_finite_adapter_reaches_its_own_tokens_only():
    import torch
    w = workload(6, 100, 264, 392, 16, 12)
    want, bad = oracle_of(w), np.isin(w.ids, [2, 7])
    w.adapters[2].B[:, 3], w.adapters[7].B[:, 0] = 0x7F80, 0x7FC0
    pool = make_pool(w)
    try:
        got = from_dev_bf16(pool.linear(to_dev_bf16(w.W), to_dev_bf16(w.x), torch.from_numpy(w.ids).cuda()))
        assert_parity(got[~bad], want[~bad], "tokens on finite adapters and on none")
        assert not np.isfinite(got[bad]).any()
    finally:
        pool.close()


@pytest.mark.parametrize("h_in,h_out,T,slots,rank", [
    (664, 864, 226, 40, 16),        # few adapters with many tokens each: their tokens count too
    (344, 344, 202, 38, 64),        # as many CTAs as K blocks
    (5216, 11224, 65, 254, 64),     # more row tiles than clusters of two: nothing is gained by a second wave
    (9440, 6184, 142, 12, 16),
])
def test_the_count_of_parts_taken(h_in, h_out, T, slots, rank):
    # every row tile's cluster is resident at once, and the count leaves no SM empty that another whole part could use where K or
    # the expand is long
    n_tiles, held = -(-h_out // 128), {1: 148, 2: 74, 3: 45, 4: 33, 5: 26, 6: 22, 7: 15, 8: 15}
    import torch
    pool = B.Pool(h_in, h_out, slots, rank, max_tokens=T)   # (no adapter loaded: the host knows no more than the slots)
    try:
        dev = lambda *shape: torch.zeros(shape, dtype=torch.bfloat16, device="cuda")
        pool.linear(dev(h_out, h_in), dev(T, h_in), torch.full((T,), -1, dtype=torch.int32, device="cuda"))
        got = B.edgelora_pool_last_launch(pool.handle)["split_k"]
        assert pool.status() == (0, 0)
    finally:
        pool.close()
    assert n_tiles <= held[got]
    if n_tiles > 74:
        assert got == 1
    else:
        assert got > 1 and (got >= 5 or n_tiles > held[got + 1])


@pytest.mark.parametrize("items", [0, 60, 20000])
def test_sums_of_k_chunks_for_all_counts_of_tokens(items):
    # groups around the four tokens and the sixteen of a round of loads, few and many K chunks (8192: 32 steps)
    counts = [1, 3, 4, 5, 15, 16, 17, 32, 33, 47]
    ids = np.random.Generator(np.random.PCG64(9)).permutation(np.repeat(np.arange(len(counts)), counts))
    w = workload(8, len(ids), 8192, 136, 32, len(counts), ids)
    y = run_gpu(w, 1, options={B.OPT_SHRINK_ITEMS: items})
    assert_parity(y, oracle_of(w), w.name)
