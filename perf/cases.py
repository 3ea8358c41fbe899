"""Performance cases of the join library: what a user's program has it do.

A case is a dict of plain values with a ``kind``:

- ``lookup``:  ``eiger.join`` of a probe column against unique build keys. The
  pairs come in unspecified order, so the program scatters them into the table
  it wants: the build row of every probe row (-1 where none matches).
- ``sum``:     ``eiger.join_sum``, the exact sum of both sides' payloads over
  all matches (foreign-key and many-to-many joins).
- ``query``:   ``eiger.join_wide`` of a fact table with a dimension (two payload
  columns a side), the joined rows then grouped by a dimension attribute with
  ``eiger.groupby`` and the groups ordered by key.
- ``groupby``: ``eiger.groupby`` with the groups ordered by key.
- ``batch``:   ``eiger.BatchedJoin.run``, many independent joins in one call,
  the pairs scattered into one row table per join as in ``lookup``.
- ``profile``: ``eiger.stats`` of a key column.

Inputs are drawn on the GPU from the seed alone.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_04489_gb300 import eiger
from paper_2607_04489_gb300.workloads import permutation, uniform_ints

DEV = "cuda"
_MAX_LOOKUP = 1 << 27  # probe rows of a drawn lookup
_MAX_SUM = 600_000_000  # probe rows of a drawn sum


# ------------------------------------------------------------------ the cases

def _lookup(nb, np_, dtype, keys, theta=0.0, absent=0.0):
    return {"kind": "lookup", "nb": nb, "np": np_, "dtype": dtype, "keys": keys, "theta": theta, "absent": absent}


def _sum(nb, np_, dtype, keys, pay, theta=0.0, absent=0.0, distinct=1.0):
    return {"kind": "sum", "nb": nb, "np": np_, "dtype": dtype, "keys": keys, "pay": pay, "theta": theta,
            "absent": absent, "distinct": distinct}


def _query(nb, np_, dtype, groups, absent):
    return {"kind": "query", "nb": nb, "np": np_, "dtype": dtype, "groups": groups, "absent": absent}


def _groupby(n, groups, dtype, aggs, theta=0.0):
    return {"kind": "groupby", "n": n, "groups": groups, "dtype": dtype, "aggs": aggs, "theta": theta}


def _batch(k, lo, hi, dtype, theta):
    return {"kind": "batch", "k": k, "log2_lo": lo, "log2_hi": hi, "dtype": dtype, "theta": theta}


def _profile(n, dtype, log2_span):
    return {"kind": "profile", "n": n, "dtype": dtype, "log2_span": log2_span}


def listed():
    return [
        # a handful of rows against a code table: launches, readbacks and host work are all there is
        dict(_lookup(1_000, 5_003, "int32", "dense"), name="lookup_tiny"),
        # the small static join of the benchmark and tests: the table stays in L2
        dict(_lookup(1 << 20, 1 << 22, "int32", "dense"), name="lookup_small"),
        # surrogate 64-bit keys (hashes, UUID halves) that do not narrow, a tenth of the probes without a partner
        dict(_lookup(5_000_011, 20_000_003, "int64", "random", absent=0.1), name="lookup_int64_random"),
        # a skewed fact column: a few hot keys take most probes
        dict(_lookup(16_000_057, 64_000_009, "int64", "dense", theta=1.0), name="lookup_skewed"),
        # a dense 64-bit surrogate key that narrows to 32 bits, the table beyond half of L2
        dict(_lookup(7_000_003, 28_000_013, "int64", "dense"), name="lookup_dense"),
        # star schema: 600M facts against a 150M-row dimension, a tenth of them dangling, both payloads summed
        dict(_sum(150_000_000, 600_000_000, "int32", "dense", "int64", absent=0.1), name="sum_star"),
        # many-to-many join on a repeated 64-bit key (about six build rows per key)
        dict(_sum(8_000_009, 30_000_001, "int64", "random", "int32", theta=0.5, distinct=0.16), name="sum_many"),
        # join, then group by an attribute of the dimension: the shape of a reporting query
        dict(_query(10_000_019, 120_000_007, "int32", 25_000, 0.05), name="query_wide"),
        # aggregation into few groups (a status, a day, a region)
        dict(_groupby((1 << 27) + 77, 3_000, "int32", "sum32,max32"), name="groupby_few"),
        # aggregation per customer or item: as the benchmark's, 2^28 rows, 4-byte keys and values
        dict(_groupby(1 << 28, 1 << 22, "int32", "sum32,max32"), name="groupby_many"),
        # thousands of small and medium joins (per shard, per tenant) in one call
        dict(_batch(4096, 6.0, 16.0, "int32", 1.0), name="batch_mixed"),
        # statistics of a column before it is planned for
        dict(_profile((1 << 27) + 5, "int64", 45), name="profile_column"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["lookup", "lookup", "lookup", "sum", "sum", "query", "groupby", "groupby", "batch", "profile"])
    dtype = rng.choice(["int32", "int64"])
    theta = rng.choice([0.0, round(rng.uniform(0.1, 1.5), 2)])
    absent = rng.choice([0.0, round(rng.uniform(0.01, 0.6), 2)])
    keys = rng.choice(["dense", "random"])
    if kind == "lookup":
        nb = _log_int(rng, 500, 1 << 25)
        return _lookup(nb, min(int(nb * rng.uniform(1, 16)), _MAX_LOOKUP), dtype, keys, theta, absent)
    if kind == "sum":
        nb = _log_int(rng, 4_000, 150_000_000)
        distinct = rng.choice([1.0, round(rng.uniform(0.1, 0.9), 2)])
        top = _MAX_SUM if distinct == 1.0 else 100_000_000
        return _sum(min(nb, top), min(int(nb * rng.uniform(0.1, 12)) + 1, top), dtype, keys,
                    rng.choice(["int32", "int64"]), min(theta, 1.0), absent, distinct)
    if kind == "query":
        nb = _log_int(rng, 1_000, 30_000_000)
        return _query(nb, min(int(nb * rng.uniform(1, 16)), 200_000_000), dtype, min(_log_int(rng, 5, 200_000), nb // 64), absent)
    if kind == "groupby":
        n = _log_int(rng, 20_000, 1 << 28)
        aggs = rng.choice(["sum32,max32", "sum64,count", "min64", "sum32,sum64,min32,count"])
        if n > 1 << 27 and aggs == "sum32,sum64,min32,count":
            n >>= 1
        return _groupby(n, _log_int(rng, 4, min(n, 1 << 24)), dtype, aggs, min(theta, 1.2))
    if kind == "batch":
        lo = round(rng.uniform(5, 11), 2)
        hi = round(lo + rng.uniform(1, 7), 2)
        mean = (2**hi - 2**lo) / ((hi - lo) * math.log(2))
        return _batch(min(_log_int(rng, 64, 16384), int(6e7 / mean) + 1), lo, hi, dtype, min(theta, 1.0))
    return _profile(_log_int(rng, 5_000, 1 << 28), dtype, rng.randint(8, 31 if dtype == "int32" else 62))


# ------------------------------------------------------------------ inputs

def _seeds(seed):
    """Independent stream seeds of one case seed."""
    n = 0
    while True:
        yield (int(seed) * 1_000_003 + n * 7919) & 0x7FFFFFFFFFFF
        n += 1


def _dtype(name):
    return torch.int32 if name == "int32" else torch.int64


def _wrap32(t):
    """int64 values modulo 2^32 as int32."""
    t = t & 0xFFFFFFFF
    return torch.where(t >= 1 << 31, t - (1 << 32), t).to(torch.int32)


def _unique_keys(n, dtype, keys, s):
    """n unique keys in random order, and a function giving keys of the same
    shape for the ids n, n + 1, ... (absent ones)."""
    p = permutation(n, next(s), DEV)
    if keys == "dense":
        lim = (1 << 40) if dtype == "int64" else (1 << 20)
        base = int(uniform_ints(1, -lim, lim, next(s))[0])
        make = lambda i: (i + base).to(_dtype(dtype))
    elif dtype == "int32":  # an affine bijection of 32 bits
        mul = int(uniform_ints(1, 0, 1 << 30, next(s))[0]) * 2 + 1
        make = lambda i: _wrap32(i * mul + 12345)
    else:  # spread over 64 bits, unique by the low bits
        bits = max(1, (2 * n - 1).bit_length())
        lim = 1 << (63 - bits)
        mul = int(uniform_ints(1, 0, 1 << 30, next(s))[0]) * 2 + 1
        make = lambda i: ((i * mul) * 2654435761 % (2 * lim) - lim) * (1 << bits) + i
    return make(p), make


def _pick(n, theta, count, s):
    """count rows of n: uniform, or skewed by the continuous power law
    (x + 1)^-theta (an approximation of Zipf's, in closed form, so that a seed
    gives the same rows every time) over a random order."""
    if theta == 0.0:
        return uniform_ints(count, 0, n, next(s), DEV)
    g = torch.Generator(device=DEV)
    g.manual_seed(next(s))
    x = torch.rand(count, generator=g, device=DEV, dtype=torch.float64)
    e = 1.0 - theta
    if abs(e) < 1e-9:
        x.mul_(math.log(n + 1.0)).exp_()
    else:
        x.mul_((n + 1.0) ** e - 1.0).add_(1.0).pow_(1.0 / e)
    return permutation(n, next(s), DEV)[x.sub_(1.0).to(torch.int64).clamp_(0, n - 1)]


def _probe_keys(bk, make, nb, np_, theta, absent, s):
    pk = bk[_pick(nb, theta, np_, s)]
    if absent > 0:
        g = torch.Generator(device=DEV)
        g.manual_seed(next(s))
        miss = torch.rand(np_, generator=g, device=DEV) < absent
        other = make(uniform_ints(np_, nb, 2 * nb, next(s), DEV))
        pk = torch.where(miss, other, pk)
    return pk


def _values(n, dtype, s):
    big = (1 << 62) if dtype == "int64" else (1 << 30)
    return uniform_ints(n, -big, big, next(s), DEV).to(_dtype(dtype))


def _batch_inputs(case, seed):
    """Flat columns of k joins: build keys, probe keys and their sizes; every
    probe row has one partner in its own join (skewed towards the first rows of
    a shuffled order by a power law)."""
    s = _seeds(seed)
    k, lo, hi = case["k"], case["log2_lo"], case["log2_hi"]
    rng = np.random.default_rng(k)  # the joins' sizes belong to the case
    nb = np.floor(2.0 ** rng.uniform(lo, hi, k)).astype(np.int64)
    npr = 4 * nb
    nbt, npt = torch.from_numpy(nb).to(DEV), torch.from_numpy(npr).to(DEV)
    boff, poff = torch.cumsum(nbt, 0) - nbt, torch.cumsum(npt, 0) - npt
    mul = torch.from_numpy(rng.integers(0, 1 << 31, k) * 2 + 1).to(DEV)
    add = torch.from_numpy(rng.integers(0, 1 << 32, k)).to(DEV)
    exp = torch.from_numpy(1.0 / (1.0 - 0.9 * rng.uniform(0, case["theta"], k) if case["theta"] else np.ones(k))).to(DEV)
    jb, jp = torch.repeat_interleave(nbt), torch.repeat_interleave(npt)
    i = torch.arange(int(nb.sum()), device=DEV) - boff[jb]
    key = i * mul[jb] + add[jb]
    key = _wrap32(key) if case["dtype"] == "int32" else key * 0x9E3779B1
    g = torch.Generator(device=DEV)
    g.manual_seed(next(s))
    u = torch.rand(int(npr.sum()), generator=g, device=DEV, dtype=torch.float64)
    n = nbt[jp]
    row = torch.minimum((u ** exp[jp] * n).to(torch.int64), n - 1)
    row = (row * 7919 + 13) % n if case["theta"] else row  # hot rows lie anywhere in the build column
    return key, key[boff[jp] + row], nb, npr, poff[jp]


def prepare(case, seed):
    s = _seeds(seed)
    kind = case["kind"]
    if kind == "lookup":
        bk, make = _unique_keys(case["nb"], case["dtype"], case["keys"], s)
        pk = _probe_keys(bk, make, case["nb"], case["np"], case["theta"], case["absent"], s)
        return {"kind": kind, "bk": bk, "pk": pk}
    if kind == "sum":
        nb, np_ = case["nb"], case["np"]
        ndv = max(1, int(nb * case["distinct"]))
        vals, make = _unique_keys(ndv, case["dtype"], case["keys"], s)
        bk = vals if ndv == nb else vals[uniform_ints(nb, 0, ndv, next(s), DEV)]
        pk = _probe_keys(vals, make, ndv, np_, case["theta"], case["absent"], s)
        return {"kind": kind, "bk": bk, "pk": pk, "bp": _values(nb, case["pay"], s), "pp": _values(np_, case["pay"], s)}
    if kind == "query":
        nb, np_ = case["nb"], case["np"]
        bk, make = _unique_keys(nb, case["dtype"], "dense", s)
        pk = _probe_keys(bk, make, nb, np_, 0.0, case["absent"], s)
        attr = uniform_ints(nb, 0, case["groups"], next(s), DEV).to(torch.int32)
        price = uniform_ints(nb, 0, 1 << 20, next(s), DEV).to(torch.int32)
        amount = uniform_ints(np_, 0, 1 << 20, next(s), DEV).to(torch.int32)
        day = uniform_ints(np_, 0, 4000, next(s), DEV).to(torch.int32)
        return {"kind": kind, "bk": bk, "pk": pk, "bc": [attr, price], "pc": [amount, day], "groups": case["groups"]}
    if kind == "groupby":
        n, g = case["n"], case["groups"]
        ids = permutation(g, next(s), DEV) * 3
        if case["dtype"] == "int64":
            ids = ids * ((1 << 38) + 1)  # spans more than 32 bits
        ids = ids.to(_dtype(case["dtype"]))
        key = ids[_pick(g, case["theta"], n, s)]
        key[torch.arange(g, device=DEV) * (n // g)] = ids  # every group has a row
        aggs = []
        for a in case["aggs"].split(","):
            op = a.rstrip("0123456789")
            aggs.append((op, None if op == "count" else _values(n, "int64" if a.endswith("64") else "int32", s)))
        return {"kind": kind, "key": key, "aggs": aggs, "groups": g}
    if kind == "batch":
        bk, pk, nb, npr, base = _batch_inputs(case, seed)
        knobs = None if case["dtype"] == "int32" else eiger.BatchKnobs()  # the stored knobs are for int32 keys
        bj = eiger.BatchedJoin(list(torch.split(bk, nb.tolist())), list(torch.split(pk, npr.tolist())), knobs=knobs)
        return {"kind": kind, "batch": bj, "base": base.to(torch.int32)}
    span = 1 << case["log2_span"]
    lo = int(uniform_ints(1, -span, max(1 - span, 1), next(s))[0]) if case["log2_span"] < 31 else -(span >> 1)
    return {"kind": kind, "key": uniform_ints(case["n"], lo, lo + span, next(s), DEV).to(_dtype(case["dtype"]))}


# ------------------------------------------------------------------ one pass

def _by_key(r):
    """The groups in key order."""
    key, order = torch.sort(r.keys)
    return {"key": key, "aggs": [a[order] for a in r.aggs]}


def run(state):
    kind = state["kind"]
    if kind == "lookup":
        r = eiger.join(state["bk"], state["pk"])
        row = torch.full((state["pk"].numel(),), -1, dtype=torch.int32, device=DEV)
        row[r.probe_idx] = r.build_idx
        return {"row": row, "count": r.count}
    if kind == "sum":
        total, count, _ = eiger.join_sum(state["bk"], state["bp"], state["pk"], state["pp"])
        return {"sum": total, "count": count}
    if kind == "query":
        j = eiger.join_wide(state["bk"], state["pk"], state["bc"], state["pc"], indices=False)
        attr, price = j.build_cols
        amount, day = j.probe_cols
        return _by_key(eiger.groupby(attr, [("sum", amount), ("max", price), ("min", day), ("count", None)],
                                     capacity=state["groups"]))
    if kind == "groupby":
        return _by_key(eiger.groupby(state["key"], state["aggs"], capacity=state["groups"]))
    if kind == "batch":
        bj = state["batch"]
        bj.run()
        row = torch.full(state["base"].shape, -1, dtype=torch.int32, device=DEV)
        row[state["base"] + bj.out_pidx] = bj.out_bidx
        return {"row": row, "counts": bj.counts, "status": bj.status}
    st = eiger.stats(state["key"])
    return {"min": st.min, "max": st.max, "estimate": st.estimate, "hll": st.hll}


def _width(dtype):
    return 4 if dtype.endswith("32") else 8


def work(case):
    """Bytes a pass cannot do without: every input column once, the call's
    outputs once (8 bytes a pair) and the row tables or ordered groups once."""
    kind = case["kind"]
    if kind == "lookup":
        kb, m = _width(case["dtype"]), case["np"] * (1 - case["absent"])
        b = kb * (case["nb"] + case["np"]) + 8 * m + 4 * case["np"]
    elif kind == "sum":
        b = (_width(case["dtype"]) + _width(case["pay"])) * (case["nb"] + case["np"])
    elif kind == "query":
        m = case["np"] * (1 - case["absent"])
        b = (_width(case["dtype"]) + 8) * (case["nb"] + case["np"]) + 16 * m + 36 * case["groups"]
    elif kind == "groupby":
        cols = [a for a in case["aggs"].split(",") if a != "count"]
        out = _width(case["dtype"]) + 8 * len(case["aggs"].split(","))
        b = (_width(case["dtype"]) + sum(_width(a) for a in cols)) * case["n"] + 2 * out * min(case["groups"], case["n"])
    elif kind == "batch":
        lo, hi = case["log2_lo"], case["log2_hi"]
        rows = case["k"] * (2**hi - 2**lo) / ((hi - lo) * math.log(2))
        b = _width(case["dtype"]) * 5 * rows + (8 + 4) * 4 * rows
    else:
        b = _width(case["dtype"]) * case["n"]
    return {"bytes": b, "flops": 0}


# ------------------------------------------------------------------ expected results

def _find(bk, pk):
    """First build row of each probe key by sorted search (-1: none)."""
    key, order = torch.sort(bk)
    at = torch.searchsorted(key, pk).clamp_(max=bk.numel() - 1)
    return torch.where(key[at] == pk, order[at], -1)


def _aggregate(key, aggs):
    u, inv = torch.unique(key, return_inverse=True)
    out = []
    for op, v in aggs:
        if op == "count":
            out.append(torch.bincount(inv, minlength=u.numel()))
        elif op == "sum":
            out.append(torch.zeros_like(u, dtype=torch.int64).scatter_add_(0, inv, v.long()))
        else:
            z = torch.zeros_like(u, dtype=torch.int64)
            out.append(z.scatter_reduce_(0, inv, v.long(), "amin" if op == "min" else "amax", include_self=False))
    return {"key": u, "aggs": out}


def _sketch(key):
    """Registers and estimate of a 2^14-register HyperLogLog over SplitMix64."""
    shr = lambda z, n: (z >> n) & ((1 << (64 - n)) - 1)
    reg = torch.zeros(1 << 14, dtype=torch.int64, device=key.device)
    for part in key.split(1 << 24):
        z = part.long()
        z = (z ^ shr(z, 30)) * (0xBF58476D1CE4E5B9 - (1 << 64))
        z = (z ^ shr(z, 27)) * (0x94D049BB133111EB - (1 << 64))
        z = z ^ shr(z, 31)
        rank = 51 - torch.frexp((z & ((1 << 50) - 1)).double()).exponent.long()
        reg.scatter_reduce_(0, shr(z, 50), rank, "amax")
    m = float(reg.numel())
    est = 0.7213 / (1 + 1.079 / m) * m * m / float(torch.exp2(-reg.double()).sum())
    zeros = int((reg == 0).sum())
    if zeros and est <= 2.5 * m:
        est = m * math.log(m / zeros)
    return reg.to(torch.uint8), est


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        bk, pk, nb, npr, _ = _batch_inputs(case, seed)
        nbt, npt = torch.from_numpy(nb).to(DEV), torch.from_numpy(npr).to(DEV)
        if case["dtype"] == "int32":  # one search over (join, key)
            jb, jp = torch.repeat_interleave(nbt), torch.repeat_interleave(npt)
            row = _find((jb << 32) + bk, (jp << 32) + pk) - (torch.cumsum(nbt, 0) - nbt)[jp]
            return {"row": row.to(torch.int32), "counts": npt, "status": torch.zeros(1, dtype=torch.int32)}
        rows = [_find(b, p) for b, p in zip(torch.split(bk, nb.tolist()), torch.split(pk, npr.tolist()))]
        return {"row": torch.cat(rows).to(torch.int32), "counts": npt, "status": torch.zeros(1, dtype=torch.int32)}
    s = prepare(case, seed)
    if kind == "lookup":
        row = torch.cat([_find(s["bk"], p) for p in s["pk"].split(1 << 28)]).to(torch.int32)
        return {"row": row, "count": int((row >= 0).sum())}
    if kind == "sum":
        key, order = torch.sort(s["bk"])
        acc = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(s["bp"][order].long(), 0)])
        total = count = 0
        for pk, pp in zip(s["pk"].split(1 << 26), s["pp"].split(1 << 26)):
            lo, hi = torch.searchsorted(key, pk), torch.searchsorted(key, pk, right=True)
            total += int((acc[hi] - acc[lo] + (hi - lo) * pp.long()).sum())
            count += int((hi - lo).sum())
        return {"sum": (total + (1 << 63)) % (1 << 64) - (1 << 63), "count": count}
    if kind == "query":
        row = _find(s["bk"], s["pk"])
        hit = row >= 0
        row = row[hit]
        attr, price = (c[row] for c in s["bc"])
        amount, day = (c[hit] for c in s["pc"])
        return _aggregate(attr, [("sum", amount), ("max", price), ("min", day), ("count", None)])
    if kind == "groupby":
        return _aggregate(s["key"], s["aggs"])
    hll, est = _sketch(s["key"])
    return {"min": int(s["key"].min()), "max": int(s["key"].max()), "estimate": est, "hll": hll.cpu().numpy()}
