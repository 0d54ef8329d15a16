"""Cases by which the speed of this framework is judged: what a program that trains or serves on the store has it do.

Every case goes through `binding.Store` as a user's program does.  `kind` says which part of the path it takes:

  pull      row lookups of a batch of keys
  push      additive updates of a batch of keys, then the replica merge (fast or ordered mode)
  round     one trainer round on a store with an accumulator table: pull both tables' rows, push updates to both, merge
  sample    PrepareSample, then PullSample of its keys and rows in one or several parts
  sgns      skip-gram steps with negative sampling
  complex   ComplEx + AdaGrad steps
  mf        matrix-factorization steps
  choose    count a stretch of the access stream, choose the hot keys anew, set their management

Sizes are those of the workloads in bench.py and of the tests, with tables of at most 20M rows so that several stores fit
one GPU; every table of a throughput case is far larger than the L2 cache.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2104_00501_b200 import binding, inputs

LEVELS = {"CONFORM": binding.CONFORM, "BOUNDED": binding.BOUNDED, "LONG-TERM": binding.LONGTERM, "NON-CONFORM": binding.NONCONFORM}
WORKERS, SYNC_EVERY, POOL_USES, POOL_SIZE, WINDOW = 8, 16, 16, 250, 5
BATCHES = 4                     # key batches that a state holds and takes in turn


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------
def listed():
    return [
        # a lookup of a few rows, as an inference request makes it: nothing but latency
        {"name": "pull_few", "kind": "pull", "keys": 1_000_000, "len": 64, "bytes": 4, "n": 96, "skew": 1.0, "top": 0},
        # the parameter-server microbenchmark: a large batch of skewed keys, the most frequent ones replicated
        {"name": "pull_many", "kind": "pull", "keys": 20_000_000, "len": 128, "bytes": 4, "n": 1 << 20, "skew": 1.0, "top": 1000},
        {"name": "push_many", "kind": "push", "keys": 20_000_000, "len": 128, "bytes": 4, "n": 1 << 20, "skew": 1.0, "top": 1000,
         "ordered": False},
        # reproducible training: updates applied in item order, an odd number of rows, milder skew
        {"name": "push_ordered", "kind": "push", "keys": 2_000_000, "len": 64, "bytes": 4, "n": 200_003, "skew": 0.9, "top": 1000,
         "ordered": True},
        # a trainer outside the library that keeps AdaGrad state beside 8-byte values
        {"name": "round_adagrad_f64", "kind": "round", "keys": 1_000_000, "len": 100, "bytes": 8, "n": 50_021, "skew": 0.9, "top": 500},
        # negatives for a trainer outside the library: pooled reuse in one go; postponing, taken in four parts by a store
        # that tracks where keys are
        {"name": "sample_reuse", "kind": "sample", "keys": 20_000_000, "len": 128, "n": 1 << 20, "level": "BOUNDED", "parts": 1, "top": 1000},
        {"name": "sample_postpone", "kind": "sample", "keys": 5_000_000, "len": 128, "n": 120_000, "level": "LONG-TERM", "parts": 4, "top": 1000},
        # word vectors at full size, 64 steps per call
        {"name": "sgns_words", "kind": "sgns", "vocab": 1_000_000, "len": 300, "batch": 4096, "steps": 64, "K": 3, "level": "BOUNDED",
         "top": 20_000, "sync": SYNC_EVERY, "lr": 0.001, "ordered": False},
        # a small model trained reproducibly, one short step per call
        {"name": "sgns_ordered_small", "kind": "sgns", "vocab": 10_000, "len": 64, "batch": 256, "steps": 1, "K": 3, "level": "CONFORM",
         "top": 100, "sync": 1, "lr": 0.025, "ordered": True},
        # knowledge-graph embeddings: two tables, wide rows, ten negatives
        {"name": "complex_kge", "kind": "complex", "entities": 2_000_000, "relations": 1000, "len": 500, "bytes": 4, "batch": 8192, "K": 10,
         "ordered": False},
        # matrix factorization, cells visited column by column
        {"name": "mf_columns", "kind": "mf", "rows": 10_000_000, "cols": 1_000_000, "len": 100, "bytes": 4, "batch": 65_536, "columns": True,
         "ordered": False},
        # the hot set chosen anew from the accesses since the last choice
        {"name": "choose_hot", "kind": "choose", "keys": 11_000_000, "len": 32, "n": 4_000_000, "skew": 0.8, "top": 10_000},
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm; odd ones as often as even ones."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above."""
    kind = rng.choice(["pull", "pull", "push", "push", "round", "sample", "sample", "sgns", "sgns", "complex", "mf", "choose"])
    if kind in ("pull", "push"):
        c = {"kind": kind, "keys": _log(rng, 200_000, 20_000_000), "len": rng.choice([32, 64, 100, 128, 128, 256]), "bytes": rng.choice([4, 4, 4, 8]),
             "n": _log(rng, 64, 1 << 20), "skew": rng.choice([0.0, 0.6, 1.0, 1.4]), "top": rng.choice([0, 1000, 20_000])}
        if kind == "push":
            c["ordered"] = rng.random() < 0.4
        size = 128 * 4 / (c["len"] * c["bytes"])           # no more bytes than the listed cases have
        c["keys"] = min(c["keys"], int(20_000_000 * size))
        c["n"] = min(c["n"], int((1 << 20) * size))
        if c.get("ordered"):
            c["n"] = min(c["n"], 300_000)
        return c
    if kind == "round":
        return {"kind": kind, "keys": _log(rng, 100_000, 2_000_000), "len": rng.choice([64, 100, 250]), "bytes": rng.choice([4, 8]),
                "n": _log(rng, 256, 100_000), "skew": rng.choice([0.0, 0.9, 1.2]), "top": rng.choice([0, 500, 5000])}
    if kind == "sample":
        parts = rng.choice([1, 1, 2, 4])
        return {"kind": kind, "keys": _log(rng, 200_000, 20_000_000), "len": rng.choice([64, 100, 128]), "n": _log(rng, 1000, 1 << 18) * parts,
                "level": rng.choice(sorted(LEVELS)), "parts": parts, "top": rng.choice([0, 1000])}
    if kind == "sgns":
        ordered = rng.random() < 0.4
        return {"kind": kind, "vocab": _log(rng, 5_000, 1_000_000), "len": rng.choice([64, 100, 200, 300]), "batch": _log(rng, 100, 4096),
                "steps": rng.choice([1, 4]) if ordered else rng.choice([1, 4, 16, 64]), "K": rng.choice([3, 3, 5]),
                "level": rng.choice(["CONFORM", "BOUNDED", "LONG-TERM"]), "top": rng.choice([0, 100, 1000]), "sync": rng.choice([1, SYNC_EVERY]),
                "lr": 0.001, "ordered": ordered}
    if kind == "complex":
        return {"kind": kind, "entities": _log(rng, 50_000, 2_000_000), "relations": 1000, "len": rng.choice([100, 200, 256, 500]),
                "bytes": rng.choice([4, 4, 8]), "batch": _log(rng, 128, 4096), "K": rng.choice([4, 10]), "ordered": rng.random() < 0.3}
    if kind == "mf":
        return {"kind": kind, "rows": _log(rng, 100_000, 5_000_000), "cols": _log(rng, 10_000, 500_000), "len": rng.choice([32, 64, 100]),
                "bytes": rng.choice([4, 4, 8]), "batch": _log(rng, 1000, 65_536), "columns": rng.random() < 0.5, "ordered": rng.random() < 0.3}
    return {"kind": kind, "keys": _log(rng, 100_000, 11_000_000), "len": 32, "n": _log(rng, 100_000, 4_000_000), "skew": rng.choice([0.8, 1.0]),
            "top": rng.choice([100, 1000, 10_000])}


# ------------------------------------------------------------------------------------------------
# what a user's program has in hand
# ------------------------------------------------------------------------------------------------
class _Table:
    """A store's table as a tensor: no copy, it shows what the table holds when it is read.  The tensor keeps this object and
    with it the store, whose memory it looks at."""

    def __init__(self, store, which):
        self.store = store
        address, stride = store.table_ptr(which)
        self.__cuda_array_interface__ = {"shape": (store.num_keys, stride), "typestr": "<f8" if store.dtype == torch.float64 else "<f4",
                                         "data": (address, False), "version": 2}


def _table(store, which=0):
    return torch.as_tensor(_Table(store, which), device=store.device)


def _i32(t):
    return t.to(torch.int32).contiguous()


def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 16 + salt)


def _key_batches(n, keys, skew, seed):
    cdf = inputs.zipf_cdf(keys, skew, "cuda") if skew else None
    return [_i32(inputs.zipf_keys(n, keys, skew, seed * BATCHES + i, "cuda", cdf=cdf)) for i in range(BATCHES)]


def _replicate_top(store, keys, top):
    """Replicate the `top` most frequent keys of the skewed streams above."""
    top = min(top, keys // 4)
    if top:
        store.set_management(_i32(inputs.rank_to_key(torch.arange(top, device="cuda"), keys, seed=1)), binding.REPLICATE)


def prepare(case, seed):
    st = {"case": case, "turn": 0}
    globals()["_prepare_" + case["kind"]](st, case, int(seed))
    return st


def _prepare_pull(st, c, seed):
    st["store"] = s = binding.Store(c["keys"], c["len"], workers=WORKERS, sync_interval=0, value_bytes=c["bytes"])
    s.init_uniform(0, seed, 0.1)
    _replicate_top(s, c["keys"], c["top"])
    st["keys"] = _key_batches(c["n"], c["keys"], c["skew"], seed)


def _prepare_push(st, c, seed):
    st["store"] = s = binding.Store(c["keys"], c["len"], workers=WORKERS, sync_interval=0, deterministic=c["ordered"], value_bytes=c["bytes"])
    s.init_uniform(0, seed, 0.1)
    _replicate_top(s, c["keys"], c["top"])
    st["keys"] = _key_batches(c["n"], c["keys"], c["skew"], seed)
    st["delta"] = torch.randn((c["n"], c["len"]), generator=_gen(seed, 1), device="cuda", dtype=s.dtype)
    st["table"] = _table(s)


def _prepare_round(st, c, seed):
    st["store"] = s = binding.Store(c["keys"], c["len"], workers=WORKERS, sync_interval=0, with_adagrad=True, value_bytes=c["bytes"])
    s.init_uniform(0, seed, 0.1)
    s.init_uniform(1, seed + 1, 0.1)
    _replicate_top(s, c["keys"], c["top"])
    st["keys"] = _key_batches(c["n"], c["keys"], c["skew"], seed)
    st["delta"] = torch.randn((c["n"], c["len"]), generator=_gen(seed, 1), device="cuda", dtype=s.dtype)
    st["delta_acc"] = st["delta"] ** 2
    st["tables"] = _table(s, 0), _table(s, 1)


def _prepare_sample(st, c, seed):
    # where keys are is tracked where the scheme asks for it
    st["store"] = s = binding.Store(c["keys"], c["len"], workers=WORKERS, sync_interval=0,
                                    track_ownership=c["level"] in ("LONG-TERM", "NON-CONFORM"))
    s.init_uniform(0, seed, 0.1)
    _replicate_top(s, c["keys"], c["top"])
    w = _i32(inputs.zipf_integer_weights(c["keys"], 1.0, "cuda"))
    st["dist"] = s.register_distribution(0, w, c["keys"], LEVELS[c["level"]], U=POOL_USES, G=POOL_SIZE, seed=seed)


def _prepare_sgns(st, c, seed):
    V, pairs = c["vocab"], c["batch"] * c["steps"]
    st["store"] = s = binding.Store(2 * V, c["len"], workers=WORKERS, sync_interval=c["sync"], deterministic=c["ordered"],
                                    track_ownership=c["level"] == "LONG-TERM")
    s.init_uniform(0, seed, 0.5 / c["len"])
    cdf = inputs.zipf_cdf(V, 1.0, "cuda")
    tokens = inputs.zipf_keys(max(2_000_000, 2 * V), V, 1.0, seed, "cuda", cdf=cdf)     # the text that the statistics come from
    s.count_accesses(_i32(tokens))
    s.count_accesses(_i32(tokens + V))
    if c["top"]:
        s.set_management(s.select_hot(True, min(c["top"], V // 4)), binding.REPLICATE)
    w = _i32(inputs.integer_weights(torch.bincount(tokens, minlength=V)))
    st["dist"] = s.register_distribution(V, w, V, LEVELS[c["level"]], U=POOL_USES, G=POOL_SIZE, seed=seed)
    centre, context = inputs.skipgram_pairs(tokens[: BATCHES * pairs // (2 * WINDOW) + 4 * WINDOW], WINDOW)
    st["pairs"] = [(_i32(centre[i * pairs:(i + 1) * pairs]), _i32(context[i * pairs:(i + 1) * pairs] + V)) for i in range(BATCHES)]
    st["loss"] = torch.zeros(c["steps"], device="cuda")
    st["table"] = _table(s)


def _prepare_complex(st, c, seed):
    E, B = c["entities"], c["batch"]
    st["store"] = s = binding.Store(E + c["relations"], c["len"], workers=WORKERS, sync_interval=SYNC_EVERY, deterministic=c["ordered"],
                                    with_adagrad=True, value_bytes=c["bytes"])
    s.init_uniform(0, seed, 0.05)
    _table(s, 1).fill_(0.1)                                # the accumulators' usual start value
    h, r, t = (_i32(x) for x in inputs.kge_triples(BATCHES * B, E, c["relations"], 0.9, 1.2, seed, "cuda"))
    s.count_accesses(torch.cat([h, t]))
    relations = torch.arange(E, E + c["relations"], device="cuda", dtype=torch.int32)
    s.set_management(torch.cat([relations, s.select_hot(False, 100)[:2000]]).contiguous(), binding.REPLICATE)
    st["dist"] = s.register_distribution(0, None, E, binding.CONFORM, seed=seed)
    st["triples"] = [tuple(x[i * B:(i + 1) * B] for x in (h, r, t)) for i in range(BATCHES)]
    st["loss"] = torch.zeros(1, device="cuda")
    st["tables"] = _table(s, 0), _table(s, 1)


def _prepare_mf(st, c, seed):
    M, N, B = c["rows"], c["cols"], c["batch"]
    st["store"] = s = binding.Store(M + N, c["len"], workers=WORKERS, sync_interval=SYNC_EVERY, deterministic=c["ordered"], value_bytes=c["bytes"])
    s.init_uniform(0, seed, 0.3)
    i, j, x = inputs.mf_cells(BATCHES * B, M, N, 0.8, c["len"], 0.1, seed, "cuda")
    s.count_accesses(torch.cat([_i32(i), _i32(j)]))
    hot = s.select_hot(False, 100)[:5000]
    if hot.numel():
        s.set_management(hot.contiguous(), binding.REPLICATE)
    if c["columns"]:
        i, j, x = inputs.mf_cells(BATCHES * B, M, N, 0.8, c["len"], 0.1, seed, "cuda", by_column_of=100 * M)
    i, j = _i32(i), _i32(j)
    st["cells"] = [tuple(y[b * B:(b + 1) * B] for y in (i, j, x)) for b in range(BATCHES)]
    st["loss"] = torch.zeros(1, device="cuda")
    st["table"] = _table(s)


def _prepare_choose(st, c, seed):
    st["store"] = binding.Store(c["keys"], c["len"], workers=WORKERS, sync_interval=0)
    st["keys"] = _key_batches(c["n"], c["keys"], c["skew"], seed)
    st["hot"] = None


# ------------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------------
def run(st):
    i = st["turn"] % BATCHES
    st["turn"] += 1
    return globals()["_run_" + st["case"]["kind"]](st, st["case"], st["store"], i)


def _run_pull(st, c, s, i):
    return s.pull(st["keys"][i])


def _run_push(st, c, s, i):
    s.push(st["keys"][i], st["delta"])
    s.sync()
    return st["table"]


def _run_round(st, c, s, i):
    values, accumulators = s.pull(st["keys"][i], with_acc=True)
    s.push(st["keys"][i], st["delta"], st["delta_acc"])
    s.sync()
    return values, accumulators, st["tables"]


def _run_sample(st, c, s, i):
    h = s.prepare_sample(st["dist"], c["n"])
    return [s.pull_sample(h, c["n"] // c["parts"]) for _ in range(c["parts"])]


def _run_sgns(st, c, s, i):
    centre, context = st["pairs"][i]
    if c["steps"] == 1:
        s.step_sgns(centre, context, st["dist"], c["K"], c["lr"], st["loss"])
    else:
        s.run_sgns(centre, context, c["batch"], st["dist"], c["K"], c["lr"], st["loss"])
    return st["loss"], st["table"]


def _run_complex(st, c, s, i):
    h, r, t = st["triples"][i]
    s.step_complex(h, r, t, st["dist"], c["K"], 0.1, 1e-10, st["loss"])
    return st["loss"], st["tables"]


def _run_mf(st, c, s, i):
    rows, cols, x = st["cells"][i]
    s.step_mf(rows, cols, x, 1e-4, 0.01, st["loss"], by_column=c["columns"])
    return st["loss"], st["table"]


def _run_choose(st, c, s, i):
    s.count_accesses(st["keys"][i])
    hot = s.select_hot(True, c["top"])
    if st["hot"] is not None:
        s.set_management(st["hot"], binding.SINGLE)
    s.set_management(hot, binding.REPLICATE)
    st["hot"] = hot
    return hot, s.hot_keys(), s.counts()


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without, and how close two correct implementations come
# ------------------------------------------------------------------------------------------------
def _distinct(n, keys, skew):
    """Expected number of distinct keys among n draws from Zipf(skew) over `keys` ranks."""
    edges = np.unique(np.concatenate([np.arange(1, min(keys, 4096) + 2), np.geomspace(1, keys + 1, 4000).astype(np.int64)])).astype(np.float64)
    edges = edges[edges <= keys + 1]
    lo, width = edges[:-1], np.diff(edges)
    p = ((lo + lo + width - 1) / 2) ** -skew
    p /= (p * width).sum()
    return float((width * -np.expm1(-n * p)).sum())


def work(case):
    c = case
    k = c["kind"]
    if k in ("pull", "push"):
        row, u = c["len"] * c["bytes"], _distinct(c["n"], c["keys"], c["skew"])
        return {"bytes": 4 * c["n"] + row * c["n"] + row * u * (1 if k == "pull" else 2), "flops": 0 if k == "pull" else c["n"] * c["len"]}
    if k == "round":
        row, u = c["len"] * c["bytes"], _distinct(c["n"], c["keys"], c["skew"])
        return {"bytes": 4 * c["n"] + 2 * (2 * row * c["n"] + 2 * row * u), "flops": 2 * c["n"] * c["len"]}
    if k == "sample":
        reuse = c["level"] in ("BOUNDED", "LONG-TERM")
        draws = max(c["n"] // POOL_USES, POOL_SIZE) if reuse else c["n"]
        row = 4 * c["len"]
        return {"bytes": 16 * min(draws, c["n"]) + 4 * c["n"] + row * c["n"] + row * _distinct(draws, c["keys"], 1.0), "flops": 0}
    if k == "sgns":
        pairs = c["batch"] * c["steps"]
        tokens = pairs / (2 * WINDOW)
        negs = pairs * c["K"] / (1 if c["level"] == "CONFORM" else POOL_USES)
        u = 2 * _distinct(tokens, c["vocab"], 1.0) + _distinct(negs, c["vocab"], 0.75)
        return {"bytes": 4 * pairs * (2 + c["K"]) + 2 * 4 * c["len"] * u, "flops": 6 * pairs * (1 + c["K"]) * c["len"]}
    if k == "complex":
        u = _distinct(2 * c["batch"], c["entities"], 0.9) + _distinct(c["batch"], c["relations"], 1.2) + c["batch"] * c["K"]
        return {"bytes": 4 * c["batch"] * (3 + c["K"]) + 4 * c["len"] * c["bytes"] * u, "flops": 24 * c["batch"] * (1 + c["K"]) * c["len"]}
    if k == "mf":
        cols = max(1.0, c["batch"] * c["cols"] / (100.0 * c["rows"])) if c["columns"] else _distinct(c["batch"], c["cols"], 0.8)
        u = _distinct(c["batch"], c["rows"], 0.8) + cols
        return {"bytes": 12 * c["batch"] + 2 * c["len"] * c["bytes"] * u, "flops": 10 * c["batch"] * c["len"]}
    # choose: the keys, their counters read and written, the counters read once, the counters handed out, the two hot lists
    return {"bytes": 4 * c["n"] + 16 * _distinct(c["n"], c["keys"], c["skew"]) + 16 * c["keys"] + 8 * c["top"], "flops": 0}


def tolerance(case):
    k = case["kind"]
    if k in ("pull", "sample", "choose") or (k == "push" and case["ordered"]):
        return "exact"                                      # copies, whole numbers, and sums whose order is fixed
    wide = case.get("bytes", 4) == 8
    if k in ("push", "round"):                              # sums in any order; 32-bit: measured up to 1e-6 (5e-6 where 400k rows meet)
        return {"rel": 1e-14, "max": 1e-12} if wide else {"rel": 1e-5, "max": 2e-3}
    if case["ordered"]:                                     # every item sees the values from before the step; 32-bit arithmetic
        return {"rel": 1e-5, "max": 1e-3}
    # Fast mode: the items of a step race, and an item may or may not see what another one added.  The largest effect that can
    # have is the distance to the ordered mode, where no item sees another's update; measured at the listed sizes: 1.2e-5
    # (largest single value 0.017), 5e-4 (0.038: the first AdaGrad steps are long whatever the gradient), 7e-5 (1e-4).
    return {"sgns": {"rel": 5e-5, "max": 0.07}, "complex": {"rel": 1.5e-3, "max": 0.15}, "mf": {"rel": 3e-4, "max": 1e-3}}[k]


# ------------------------------------------------------------------------------------------------
# the same results in 64 bits, without the framework
# ------------------------------------------------------------------------------------------------
def _start_values(keys, length, seed, which, scale):
    """The start values of a table (uniform in [-scale, scale)), from the published generator: Philox4x32-10 with the counter
    (block of four values, table, 3) and the seed as its key; 24 bits of a word make a value."""
    out = torch.empty(keys * length, dtype=torch.float64, device="cuda")
    unit = float(np.float32(scale) * np.float32(1.0 / 8388608.0))
    low, step = 0xFFFFFFFF, 1 << 26

    def product(a, b):                                      # high and low half of a 32 x 32-bit product, in 64-bit integers
        lo = a * (b & 0xFFFF)
        hi = a * (b >> 16) + (lo >> 16)
        return hi >> 16, ((hi & 0xFFFF) << 16) | (lo & 0xFFFF)

    for first in range(0, out.numel() // 4, step):
        i = torch.arange(first, min(first + step, out.numel() // 4), device="cuda")
        c = [i & low, i >> 32, torch.full_like(i, which), torch.full_like(i, 3)]
        k0, k1 = seed & low, (seed >> 32) & low
        for _ in range(10):
            h0, l0 = product(c[0], 0xD2511F53)
            h1, l1 = product(c[2], 0xCD9E8D57)
            c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
            k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
        words = torch.stack([(w >> 8) - 8388608 for w in c], dim=1).to(torch.float32) * unit     # rounded as the table holds it
        out[4 * first:4 * first + words.numel()] = words.reshape(-1).double()
    return out.view(keys, length)


def _keys_of(keys, n, skew, seed):
    """The first key batch of a state."""
    return inputs.zipf_keys(n, keys, skew, seed * BATCHES, "cuda", cdf=inputs.zipf_cdf(keys, skew, "cuda") if skew else None).long()


def exact(case, seed):
    """What the first pass returns, in 64 bits.  None: copies and whole numbers; steps in which items race, where any order of
    them is right; steps whose negatives come from the store's own sampler."""
    c, seed = case, int(seed)
    if c["kind"] == "push":
        table = _start_values(c["keys"], c["len"], seed, 0, 0.1)
        dtype = torch.float64 if c["bytes"] == 8 else torch.float32
        delta = torch.randn((c["n"], c["len"]), generator=_gen(seed, 1), device="cuda", dtype=dtype)
        return table.index_add_(0, _keys_of(c["keys"], c["n"], c["skew"], seed), delta.double())
    if c["kind"] == "round":
        tables = _start_values(c["keys"], c["len"], seed, 0, 0.1), _start_values(c["keys"], c["len"], seed + 1, 1, 0.1)
        keys = _keys_of(c["keys"], c["n"], c["skew"], seed)
        dtype = torch.float64 if c["bytes"] == 8 else torch.float32
        delta = torch.randn((c["n"], c["len"]), generator=_gen(seed, 1), device="cuda", dtype=dtype)
        pulled = tables[0][keys], tables[1][keys]
        tables[0].index_add_(0, keys, delta.double())
        tables[1].index_add_(0, keys, (delta ** 2).double())
        return (*pulled, tables)
    if c["kind"] == "mf" and c["ordered"]:
        M, N, B = c["rows"], c["cols"], c["batch"]
        table = _start_values(M + N, c["len"], seed, 0, 0.3)
        i, j, x = inputs.mf_cells(BATCHES * B, M, N, 0.8, c["len"], 0.1, seed, "cuda", by_column_of=100 * M if c["columns"] else 0)
        i, j, x = i[:B].long(), j[:B].long(), x[:B].double()
        rate, decay = float(np.float32(1e-4)), float(np.float32(0.01))
        w, h = table[i], table[j]
        err = x - (w * h).sum(1)
        table.index_add_(0, i, rate * (err[:, None] * h - decay * w))
        table.index_add_(0, j, rate * (err[:, None] * w - decay * h))
        return (err ** 2).mean().reshape(1), table
    return None
