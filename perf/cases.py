"""The calls by which the speed of this library is judged.

A case is one call (or one serving step of a few calls) through the public binding, on device buffers
that a server keeps: the batched LoRA layer of one linear site, a set of sites over one batch, the
router's scoring head.  A batch is described as a serving step is formed: ``decode`` tokens (one per
generating request, adapters by the bounded power law, a share ``base`` of them without an adapter),
then ``prompt_tokens`` tokens of ``prompts`` prompts, each a run of tokens on one adapter.

Values as everywhere in this repository: W, A, B ~ N(0, 0.02), x ~ N(0, 1), bfloat16, scale 2.0.
"""
import math

import numpy as np
import torch

from paper_2507_01438_b200 import binding as lib

SCALE = 2.0
STD = 0.02
ZIPF = 1.1
# Shape of one decoder layer: (input number, h_in, h_out) per projection, by the names of the widths.
LAYER = [(0, "hidden", "hidden"), (0, "hidden", "kv"), (0, "hidden", "kv"), (0, "hidden", "hidden"),
         (0, "hidden", "ffn"), (0, "hidden", "ffn"), (1, "ffn", "hidden")]


def _linear(name, h_in, h_out, slots, rank, decode=0, prompts=0, prompt_tokens=0, base=0.0, distinct=False,
            ragged=False, mixed_ranks=False, storage="bf16", swaps=0):
    return dict(name=name, kind="linear", h_in=h_in, h_out=h_out, slots=slots, rank=rank, decode=decode,
                prompts=prompts, prompt_tokens=prompt_tokens, base=base, distinct=distinct, ragged=ragged,
                mixed_ranks=mixed_ranks, storage=storage, swaps=swaps)


def _set(name, layers, hidden, kv, ffn, slots, rank, decode=0, prompts=0, prompt_tokens=0, base=0.0, ragged=False):
    return dict(name=name, kind="set", layers=layers, hidden=hidden, kv=kv, ffn=ffn, slots=slots, rank=rank,
                decode=decode, prompts=prompts, prompt_tokens=prompt_tokens, base=base, distinct=False,
                ragged=ragged, mixed_ranks=True)


def _router(name, adapters, hidden, prompts):
    return dict(name=name, kind="router", adapters=adapters, hidden=hidden, prompts=prompts)


def listed():
    return [
        # the smallest layer call: the repository's tiny configuration (launches and latency)
        _linear("tiny_T16", 256, 256, 4, 8, decode=16, base=0.2),
        # one generating request alone: the key projection of a decoder layer
        _linear("kv_decode_T1", 4096, 1024, 16, 16, decode=1, distinct=True),
        # attention projection, every generating request on an adapter of its own
        _linear("q_decode_T32", 4096, 4096, 32, 16, decode=32, distinct=True),
        # the same step while requests come and go: two adapters arrive in Q8_0 in front of it
        _linear("q_decode_T32_swaps", 4096, 4096, 32, 16, decode=32, distinct=True, swaps=2),
        # widths and a batch that fill no tile: between the small and the large decode regime
        _linear("ragged_decode_T77", 3080, 5000, 100, 32, decode=77, base=0.1, mixed_ranks=True),
        # many tenants: 1000 resident adapters, the widest input
        _linear("down_decode_T256", 14336, 4096, 1000, 64, decode=256, base=0.1),
        # the same batch with A kept in the 8-bit format in device memory
        _linear("down_decode_T256_q8", 14336, 4096, 1000, 64, decode=256, base=0.1, storage="q8"),
        # prompts only: eight of 512 tokens through the gate / up projection
        _linear("gate_prefill_T4096", 4096, 14336, 8, 16, prompts=8, prompt_tokens=4096),
        # prompts of all lengths and some generating requests, odd widths
        _linear("ragged_prefill_T1111", 3080, 5000, 64, 64, decode=23, prompts=9, prompt_tokens=1088, base=0.1,
                ragged=True, mixed_ranks=True),
        # a serving step of generation only, through the seven projections of four decoder layers
        _set("set_decode_T27", 4, 4096, 1024, 14336, 64, 32, decode=27),
        # the benchmark's serving step: 64 generating requests and two prompts of 1024 tokens
        _set("set_mixed_T2112", 4, 4096, 1024, 14336, 128, 32, decode=64, prompts=2, prompt_tokens=2048),
        # adapter choice for prompts that have just arrived: 1000 adapters
        _router("router_1000", 1000, 4096, 4),
    ]


def _spread(rng, lo, hi, step=1):
    """A multiple of step in [lo, hi], uniform over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "prefill", "prefill", "set_decode", "set_mixed", "router"])
    rank = rng.choice([8, 16, 32, 64])
    if kind == "router":
        c = _router("", _spread(rng, 50, 2000), _spread(rng, 1024, 8192, 8), _spread(rng, 1, 16))
    elif kind == "decode":
        q8 = rng.random() < 0.2
        step = 256 if q8 else 8
        slots = _spread(rng, 4, 1000)
        c = _linear("", _spread(rng, 256, 14336, step), _spread(rng, 256, 14336, 8), slots, rank,
                    decode=_spread(rng, 1, 256), base=rng.choice([0.0, 0.1]), mixed_ranks=rng.random() < 0.5,
                    storage="q8" if q8 else "bf16", swaps=0 if q8 or rng.random() < 0.8 else rng.randint(1, min(4, slots)))
        c["swaps"] = c["swaps"] if c["h_in"] % 32 == 0 else 0    # the 8-bit blocks hold 32 values of a row
    elif kind == "prefill":
        prompts = _spread(rng, 1, 32)
        c = _linear("", _spread(rng, 512, 14336, 8), _spread(rng, 512, 14336, 8), _spread(rng, 32, 256), rank,
                    decode=rng.choice([0, rng.randint(1, 64)]), prompts=prompts,
                    prompt_tokens=_spread(rng, max(257, prompts), 8192), base=rng.choice([0.0, 0.1]),
                    ragged=rng.random() < 0.7, mixed_ranks=rng.random() < 0.5)
    else:
        hidden = _spread(rng, 1024, 4096, 128)
        mixed = kind == "set_mixed"
        prompts = rng.randint(1, 4) if mixed else 0
        c = _set("", rng.randint(1, 4), hidden, hidden // rng.choice([1, 2, 4]),
                 _spread(rng, 2 * hidden, 14336, 64), _spread(rng, 16, 128), min(rank, 32),
                 decode=_spread(rng, 1, 64), prompts=prompts,
                 prompt_tokens=_spread(rng, 257, 2048) if mixed else 0, base=rng.choice([0.0, 0.1]),
                 ragged=rng.random() < 0.7)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------- inputs

def _tokens(case):
    return case["decode"] + case["prompt_tokens"]


def _power_law(n):
    p = np.arange(1, n + 1, dtype=np.float64) ** -ZIPF
    return p / p.sum()


def _adapter_ids(case, rng):
    """int32 [T]: the slot of every token's adapter, -1 for a token without one."""
    slots, n = case["slots"], case["decode"]
    if case["distinct"]:
        ids = rng.permutation(slots)[:n]
    else:
        ids = rng.permutation(slots)[rng.choice(slots, size=n, p=_power_law(slots))]
        ids[rng.choice(n, size=int(round(case["base"] * n)), replace=False)] = -1
    k, total = case["prompts"], case["prompt_tokens"]
    if k:
        if case["ragged"]:    # every prompt has a token at least
            cuts = np.sort(rng.choice(np.arange(1, total), size=k - 1, replace=False))
            lengths = np.diff(np.concatenate([[0], cuts, [total]]))
        else:
            lengths = np.full(k, total // k)
            lengths[: total % k] += 1
        who = rng.choice(slots, size=k, replace=k > slots)
        ids = np.concatenate([ids, np.repeat(who, lengths)])
    return ids.astype(np.int32)


def _ranks_of(case, rng):
    r = case["rank"]
    choice = [max(r // 4, 4), max(r // 2, 4), r] if case["mixed_ranks"] else [r]
    return rng.choice(np.array(choice), size=case["slots"]).astype(np.int64)


def _normal(gen, shape, std=1.0):
    return (torch.randn(shape, generator=gen, device="cuda") * std).to(torch.bfloat16)


def _q8_blocks(v):
    """Rows of values in Q8_0: uint8 [rows, blocks of 32, 34], a row's last block filled up with zeros."""
    rows, n = v.shape
    nb = (n + 31) // 32
    b = torch.nn.functional.pad(v.float(), (0, nb * 32 - n)).view(rows, nb, 32)
    d = (b.abs().amax(-1, keepdim=True) / 127.0).half()
    q = torch.where(d > 0, (b / d.float()).round().clamp(-127, 127), torch.zeros_like(b)).to(torch.int8)
    return torch.cat([d.view(torch.uint8), q.view(torch.uint8)], dim=-1).contiguous()


def _host_adapter(gen, rank, h_in, h_out, q8):
    """A [rank, h_in] and B [h_out, rank] on the host, as the load calls take them."""
    a, b = _normal(gen, (rank, h_in), STD), _normal(gen, (h_out, rank), STD)
    if q8:
        return _q8_blocks(a).cpu().numpy(), _q8_blocks(b).cpu().numpy()
    return (a.view(torch.int16).cpu().numpy().view(np.uint16), b.view(torch.int16).cpu().numpy().view(np.uint16))


class _Site:
    """A linear site as a server holds it: its weights, its pool and the adapters the batch touches."""

    def __init__(self, case, h_in, h_out, ids, ranks, gen, q8=False):
        self.W = _normal(gen, (h_out, h_in), STD)
        self.pool = lib.Pool(h_in, h_out, case["slots"], case["rank"], max_tokens=max(256, _tokens(case)),
                             flags=lib.FLAG_A_Q8 if q8 else 0)
        for a in np.unique(ids[ids >= 0]):
            A, B = _host_adapter(gen, int(ranks[a]), h_in, h_out, q8)
            load = lib.edgelora_pool_load_slot_q8 if q8 else lib.edgelora_pool_load_slot
            load(self.pool.handle, int(a), int(ranks[a]), SCALE, A, B)
        lib.edgelora_pool_wait_loads(self.pool.handle)


class _SiteSet:
    def __init__(self, sites, inputs, n_inputs, max_tokens):
        self.sites = sites    # the set borrows their pools and weights
        self.handle = lib.edgelora_siteset_create([s.pool.handle for s in sites], [s.W for s in sites], inputs,
                                                  n_inputs, max_tokens)

    def __del__(self):
        lib.edgelora_siteset_destroy(self.handle)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    if case["kind"] == "router":
        n, hidden, b = case["adapters"], case["hidden"], case["prompts"]
        return {"kind": "router", "Wr": _normal(gen, (n, hidden), STD), "h": _normal(gen, (b, hidden)),
                "bias": torch.randn(n, generator=gen, device="cuda"),
                "scores": torch.empty(b, n, device="cuda")}
    T = _tokens(case)
    ids, ranks = _adapter_ids(case, rng), _ranks_of(case, rng)
    state = {"kind": case["kind"], "ids": torch.from_numpy(ids).cuda()}
    if case["kind"] == "set":
        sites, inputs = [], []
        for _ in range(case["layers"]):
            for which, h_in, h_out in LAYER:
                sites.append(_Site(case, case[h_in], case[h_out], ids, ranks, gen))
                inputs.append(which)
        state["set"] = _SiteSet(sites, inputs, 2, T)
        state["x"] = [_normal(gen, (T, case["hidden"])), _normal(gen, (T, case["ffn"]))]
        state["y"] = [torch.empty(T, s.W.shape[0], dtype=torch.bfloat16, device="cuda") for s in sites]
        return state
    h_in, h_out = case["h_in"], case["h_out"]
    state["site"] = _Site(case, h_in, h_out, ids, ranks, gen, q8=case["storage"] == "q8")
    state["x"] = _normal(gen, (T, h_in))
    state["y"] = torch.empty(T, h_out, dtype=torch.bfloat16, device="cuda")
    # adapters that arrive with the step, into slots of the batch (an unloaded slot's may be among them)
    slots = rng.permutation(case["slots"])[: case["swaps"]]
    state["arrivals"] = [(int(a), int(ranks[a]), *_host_adapter(gen, int(ranks[a]), h_in, h_out, True)) for a in slots]
    return state


# ------------------------------------------------------------------------------------------------ a pass

def run(state):
    if state["kind"] == "router":
        return lib.edgelora_router_scores(state["Wr"], state["bias"], state["h"], state["scores"])
    if state["kind"] == "set":
        lib.edgelora_siteset_run(state["set"].handle, state["x"], state["ids"], state["y"])
        return state["y"]
    pool = state["site"].pool
    for slot, rank, A, B in state["arrivals"]:
        lib.edgelora_pool_load_slot_q8(pool.handle, slot, rank, SCALE, A, B)
    return pool.linear(state["site"].W, state["x"], state["ids"], state["y"])


def _touched(case):
    """Expected number of distinct adapters of a batch."""
    n = case["decode"]
    if case["distinct"]:
        return n
    n -= int(round(case["base"] * n))
    return float((1.0 - (1.0 - _power_law(case["slots"])) ** n).sum()) + min(case["prompts"], case["slots"])


def work(case):
    """W, x, y and the touched adapters once each; the operations of both products."""
    if case["kind"] == "router":
        n, hidden, b = case["adapters"], case["hidden"], case["prompts"]
        return {"bytes": 2 * hidden * (n + b) + 4 * n * (b + 1), "flops": 2 * n * hidden * b}
    T = _tokens(case)
    r = case["rank"]
    rank = sum((max(r // 4, 4), max(r // 2, 4), r)) / 3 if case["mixed_ranks"] else r
    with_adapter = T - int(round(case["base"] * case["decode"]))
    adapters = min(_touched(case), case["slots"])
    if case["kind"] == "set":
        shapes = [(case[h_in], case[h_out]) for _, h_in, h_out in LAYER] * case["layers"]
        nbytes = 2 * T * (case["hidden"] + case["ffn"])    # the two inputs that the sites share
        swapped, a_bytes = 0, 2.0
    else:
        shapes = [(case["h_in"], case["h_out"])]
        nbytes = 2 * T * case["h_in"]
        swapped, a_bytes = case["swaps"], 34 / 32 if case["storage"] == "q8" else 2.0
    flops = 0
    for h_in, h_out in shapes:
        nbytes += 2 * h_in * h_out + 2 * T * h_out + adapters * rank * (a_bytes * h_in + 2 * h_out)
        nbytes += swapped * rank * (h_in + h_out) * (34 / 32 + 2)    # read in the 8-bit form, written in bfloat16
        flops += 2 * T * h_in * h_out + 2 * with_adapter * rank * (h_in + h_out)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the distance to the same products in 64 bits: a bfloat16 result is off by 1.7e-3 of its norm (its
    rounding) and 6e-3 of a value; the scores are 32-bit sums of exact products, off by 6e-8 here, by more in another order."""
    if case["kind"] == "router":
        return {"rel": 2e-6, "max": 1e-5}
    return {"rel": 6e-3, "max": 2.5e-2}
