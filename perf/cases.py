"""The work a user of this library has it do, as cases to be timed.

A case is one pass through the public entry points on keys that are already in
GPU memory: a lookup against a resident function, or a construction followed
by queries of what was built (the function is read back through its indices,
as a caller reads it).  Key sets, gammas, layouts and set sizes are those of
the benchmark, the tests and the paper's tables: 1e6, 1e8 and (as far as three
sets of inputs fit one GPU) 1e10 keys, gamma 1 and 2 and 5, 4096 sets of 1e3 to
1e6 keys, 18-character strings, lookup batches of 1 to 1e6 keys.
"""
import math

import numpy as np
import torch

from paper_1702_03154_gb300 import mphf

LEVELS = 25


def listed():
    return [
        # a serving process answering one small request from a resident function
        {"name": "lookup_1k", "kind": "lookup", "n": 1_000_000, "q": 1_000, "gamma": 2.0,
         "layout": 32, "order": "random", "absent": 0.05, "shift": 0},
        # a coalesced batch of requests against many resident functions, some of
        # the keys unknown to them
        {"name": "multi_64", "kind": "multi", "functions": 64, "requests": 64, "nlo": 10_000,
         "nhi": 10_000_000, "blo": 1, "bhi": 1_000_000, "gamma": 2.0, "absent": 0.05},
        # the smallest sets: one of many small dictionaries, built on demand
        {"name": "build_10k", "kind": "build", "n": 10_007, "q": 1_001, "gamma": 2.0, "layout": 32,
         "order": "random", "shift": 0},
        # an ordinary set (the 1e6-key configuration)
        {"name": "build_1m", "kind": "build", "n": 1_000_000, "q": 100_000, "gamma": 2.0,
         "layout": 32, "order": "random", "shift": 0},
        # the smallest function a user can ask for: gamma 1 with the minirank
        # layout; odd size, keys that start off a 16-byte boundary, every key queried
        {"name": "build_23m_minirank", "kind": "build", "n": 23_000_011, "q": 23_000_011,
         "gamma": 1.0, "layout": 64, "order": "shuffled", "shift": 1},
        # the 1e8-key configuration
        {"name": "build_100m", "kind": "build", "n": 100_000_000, "q": 10_000_000, "gamma": 2.0,
         "layout": 32, "order": "random", "shift": 0},
        # massive sets (the path of the 1e10-key configuration)
        {"name": "build_3g", "kind": "build", "n": 3_000_000_000, "q": 300_000_000, "gamma": 2.0,
         "layout": 32, "order": "random", "shift": 0},
        # every key of the 1e8-key function in shuffled order (function in L2)
        {"name": "lookup_100m", "kind": "lookup", "n": 100_000_000, "q": 100_000_000, "gamma": 2.0,
         "layout": 32, "order": "shuffled", "absent": 0.0, "shift": 0},
        # bulk queries against a function far larger than L2
        {"name": "lookup_hbm", "kind": "lookup", "n": 2_000_000_000, "q": 100_000_001, "gamma": 2.0,
         "layout": 32, "order": "random", "absent": 0.0, "shift": 0},
        # a thousand key sets built together and queried
        {"name": "batched_1000", "kind": "batched", "sets": 1_000, "nlo": 1_000, "nhi": 1_000_000,
         "gamma": 2.0},
        # the partitioned form, all parts on one GPU
        {"name": "partitioned_400m", "kind": "partitioned", "n": 400_000_000, "q": 100_000_000,
         "parts": 8, "gamma": 2.0},
        # byte strings (the random 18-character strings of the paper's second table)
        {"name": "strings_20m", "kind": "strings", "n": 20_000_000, "lo": 18, "hi": 18,
         "gamma": 2.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build", "build", "build", "build", "lookup", "lookup", "lookup", "multi",
                       "batched", "partitioned", "strings"])
    gamma = rng.choice([1.0, 2.0, 2.0, 2.0, 5.0])
    layout = rng.choice([32, 32, 32, 64, 8])
    order = rng.choice(["random", "shuffled"])
    shift = rng.choice([0, 0, 1])
    if kind == "build":
        n = _log(rng, 1_000, 1_000_000_000)
        q = n if order == "shuffled" else max(1, n // rng.randint(4, 16))
        return {"kind": kind, "n": n, "q": q, "gamma": gamma, "layout": layout, "order": order,
                "shift": shift}
    if kind == "lookup":
        n = _log(rng, 10_000, 1_500_000_000)
        q = n if order == "shuffled" and n <= 200_000_000 else _log(rng, 1, 100_000_000)
        order = "shuffled" if q == n else "random"
        return {"kind": kind, "n": n, "q": q, "gamma": gamma, "layout": layout, "order": order,
                "absent": rng.choice([0.0, 0.0, 0.05, 0.5]), "shift": shift}
    if kind == "multi":
        return {"kind": kind, "functions": _log(rng, 2, 256), "requests": _log(rng, 2, 512),
                "nlo": 10_000, "nhi": _log(rng, 100_000, 10_000_000), "blo": 1,
                "bhi": _log(rng, 1_000, 1_000_000), "gamma": gamma,
                "absent": rng.choice([0.0, 0.05])}
    if kind == "batched":
        return {"kind": kind, "sets": _log(rng, 16, 4_096), "nlo": _log(rng, 1, 5_000),
                "nhi": _log(rng, 20_000, 1_000_000), "gamma": gamma}
    if kind == "partitioned":
        n = _log(rng, 1_000_000, 500_000_000)
        return {"kind": kind, "n": n, "q": max(1, n // rng.randint(2, 8)),
                "parts": rng.choice([2, 3, 4, 8, 16, 64]), "gamma": gamma}
    lo = rng.randint(16, 24)
    return {"kind": "strings", "n": _log(rng, 10_000, 30_000_000), "lo": lo,
            "hi": lo + rng.choice([0, 0, 7, 24]), "gamma": gamma}


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _keys(n, seed, shift, start=0):
    """n distinct keys; shift = 1: a view that starts 8 bytes off a 16-byte boundary."""
    return mphf.keygen(n + shift, 1_000_003 * seed + 17, start=start)[shift:]


def _pick(keys, q, order, gen):
    """q member queries: every key once in shuffled order, or uniformly with repetition."""
    n = keys.numel()
    if order == "shuffled":
        return keys[torch.randperm(n, device="cuda", generator=gen)[:q]]
    return keys[torch.randint(0, n, (q,), device="cuda", generator=gen)]


def _with_absent(queries, share, seed, gen):
    """The same queries with about `share` of them replaced by keys of no function."""
    if share <= 0:
        return queries
    other = mphf.keygen(queries.numel(), 1_000_003 * seed + 19, start=1 << 40)
    return torch.where(torch.rand(queries.numel(), device="cuda", generator=gen) < share, other,
                       queries)


def _sizes(count, lo, hi, stream):
    """Log-uniform sizes, the same for every seed (so that outputs keep their shapes)."""
    r = np.random.Generator(np.random.PCG64(stream))
    return np.clip(np.floor(np.exp(r.uniform(math.log(lo), math.log(hi), count))), lo,
                   hi).astype(np.int64)


def prepare(case, seed):
    gen = _gen(seed)
    kind, gamma = case["kind"], case["gamma"]
    st = {"case": case, "kind": kind, "gamma": gamma, "hash_seed": seed % 1009}
    if kind == "build":
        st["keys"] = _keys(case["n"], seed, case["shift"])
        st["queries"] = _pick(st["keys"], case["q"], case["order"], gen)
    elif kind == "lookup":
        keys = _keys(case["n"], seed, 0)
        st["f"] = mphf.build(keys, gamma=gamma, levels=LEVELS, seed=st["hash_seed"])
        if case["layout"] != 32:
            st["f"].set_layout(case["layout"])
        q = _with_absent(_pick(keys, case["q"], case["order"], gen), case["absent"], seed, gen)
        st["queries"] = q if not case["shift"] else torch.cat((q[:1], q))[1:]
    elif kind == "multi":
        sizes = _sizes(case["functions"], case["nlo"], case["nhi"], 11)
        sets = [mphf.keygen(int(n), 1_000_003 * seed + 100 + i) for i, n in enumerate(sizes)]
        fs = [mphf.build(k, gamma=gamma, levels=LEVELS, seed=st["hash_seed"]) for k in sets]
        batch = _sizes(case["requests"], case["blo"], case["bhi"], 12)
        which = np.random.Generator(np.random.PCG64(seed)).integers(0, len(fs), batch.size)
        st["fs"] = [fs[i] for i in which]
        st["queries"] = [_with_absent(_pick(sets[i], int(b), "random", gen), case["absent"],
                                      seed + 3 + j, gen)
                         for j, (i, b) in enumerate(zip(which, batch))]
        st["out"] = torch.empty(int(batch.sum()), dtype=torch.int64, device="cuda")
        st["outs"] = list(torch.split(st["out"], batch.tolist()))
    elif kind == "batched":
        sizes = _sizes(case["sets"], case["nlo"], case["nhi"], 7)
        st["offsets"] = np.concatenate(([0], np.cumsum(sizes))).astype(np.uint64)
        st["keys"] = mphf.keygen(int(sizes.sum()), 1_000_003 * seed + 23)
        st["queries"] = list(torch.split(st["keys"], sizes.tolist()))
        st["out"] = torch.empty_like(st["keys"])
        st["outs"] = list(torch.split(st["out"], sizes.tolist()))
    elif kind == "partitioned":
        st["keys"] = _keys(case["n"], seed, 0)
        st["queries"] = _pick(st["keys"], case["q"], "random", gen)
    elif kind == "strings":
        n = case["n"]
        if case["lo"] == case["hi"]:
            st["offsets"] = torch.arange(n + 1, device="cuda", dtype=torch.int64) * case["lo"]
        else:
            lens = torch.randint(case["lo"], case["hi"] + 1, (n,), device="cuda", generator=gen)
            st["offsets"] = torch.zeros(n + 1, device="cuda", dtype=torch.int64)
            torch.cumsum(lens, 0, out=st["offsets"][1:])
        st["data"] = torch.randint(ord("a"), ord("z") + 1, (int(st["offsets"][-1]),),
                                   device="cuda", dtype=torch.uint8, generator=gen)
    else:
        raise ValueError(kind)
    if kind in ("build", "lookup", "partitioned"):
        st["out"] = torch.empty_like(st["queries"])
    return st


def _shape(f):
    """What a caller reads off a built function (numbers the library keeps on the host)."""
    return {"bits": f.total_bits, "levels": f.num_levels, "fallback": f.num_fallback}


def run(st):
    kind, gamma, seed = st["kind"], st["gamma"], st["hash_seed"]
    if kind == "lookup":
        return st["f"].lookup(st["queries"], out=st["out"])
    if kind == "multi":
        mphf.lookup_multi(st["fs"], st["queries"], st["outs"])
        return st["out"]
    if kind == "build":
        f = mphf.build(st["keys"], gamma=gamma, levels=LEVELS, seed=seed)
        if st["case"]["layout"] != 32:
            f.set_layout(st["case"]["layout"])
        return {"index": f.lookup(st["queries"], out=st["out"]), **_shape(f)}
    if kind == "batched":
        fs = mphf.build_batched(st["keys"], st["offsets"], gamma=gamma, levels=LEVELS, seed=seed)
        mphf.lookup_multi(fs, st["queries"], st["outs"])
        return {"index": st["out"], "bits": np.array([f.total_bits for f in fs])}
    if kind == "partitioned":
        p = mphf.PartitionedMPHF.build(st["keys"], st["case"]["parts"], 12345, gamma=gamma,
                                       levels=LEVELS, seed=seed)
        return {"index": p.lookup(st["queries"], out=st["out"]),
                "offsets": p.offsets.astype(np.int64)}
    keys = mphf.string_keys(st["data"], st["offsets"], seed=seed)
    f = mphf.build(keys, gamma=gamma, levels=LEVELS, seed=seed)
    return {"keys": keys, "index": f.lookup(keys), **_shape(f)}


def _function_bytes(n, gamma, layout=32):
    """A (gamma e^(1/gamma) bits a key) with the counts of its layout."""
    share = {32: 8 / 7, 64: 16 / 15, 8: 4 / 3}[layout]
    return n * gamma * math.exp(1 / gamma) / 8 * share


def _lookup_bytes(n, q, gamma, layout=32):
    """Queries in, indices out, and the function once, or one record a probe if
    that is less (e^(1/gamma) probes a member on average)."""
    record = {32: 32, 64: 64, 8: 8}[layout]
    return 16 * q + min(_function_bytes(n, gamma, layout), q * math.exp(1 / gamma) * record)


def _mean_size(lo, hi):
    return (hi - lo) / math.log(hi / lo) if hi > lo else lo


def work(case):
    kind, gamma = case["kind"], case["gamma"]
    if kind == "lookup":
        b = _lookup_bytes(case["n"], case["q"], gamma, case["layout"])
    elif kind == "multi":
        q = _mean_size(case["blo"], case["bhi"])
        b = case["requests"] * _lookup_bytes(_mean_size(case["nlo"], case["nhi"]), q, gamma)
    elif kind == "build":
        b = (8 * case["n"] + _function_bytes(case["n"], gamma, case["layout"])
             + _lookup_bytes(case["n"], case["q"], gamma, case["layout"]))
    elif kind == "batched":
        n = case["sets"] * _mean_size(case["nlo"], case["nhi"])
        b = 8 * n + _function_bytes(n, gamma) + _lookup_bytes(n, n, gamma)
    elif kind == "partitioned":
        b = (8 * case["n"] + _function_bytes(case["n"], gamma)
             + _lookup_bytes(case["n"], case["q"], gamma))
    else:
        n = case["n"]
        text = n * ((case["lo"] + case["hi"]) / 2 + 8)
        b = text + 8 * n + 8 * n + _function_bytes(n, gamma) + _lookup_bytes(n, n, gamma)
    return {"bytes": b, "flops": 0}


def exact(case, seed):
    """Every output is a whole number (an index, a key, a count): there is no
    rounding to measure, and they are compared bit by bit."""
    return None
