"""The fused sum of the partitioned join with carried payloads (GFTR) against
the oracle: one shared-memory table per build chunk maps each distinct key to
the sum of its payloads and its row count.

Edges: build partitions of one row, just below, at and above one table's 4608
rows (several chunks), every build row the same key, keys whose encoded pattern
is all ones (the table's empty pattern), as an offset or once mixed, payloads whose sums carry between the
32-bit halves and wrap modulo 2^64, 4- and 8-byte payloads, no match at all.
Sums are integers modulo 2^64: compared exactly.
"""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eiger():
    from paper_2607_04489_gb300 import eiger

    eiger.load()
    return eiger


def _unmixed(h, bits, a, b):
    """The value that x * a, xor with its upper half shifted down, * b (all
    modulo 2^bits) mixes to h."""
    m = (1 << bits) - 1
    y = h * pow(b, -1, 1 << bits) & m
    return (y ^ (y >> bits // 2)) * pow(a, -1, 1 << bits) & m


# keys whose offset from the type's minimum mixes to all ones
ONES32 = _unmixed(2**32 - 1, 32, 0x9E3779B1, 0x85EBCA6B) - 2**31
ONES64 = _unmixed(2**64 - 1, 64, 0x9E3779B97F4A7C15, 0xFF51AFD7ED558CCD)
ONES64 -= 2**63


def _keys(kind, rng, nb, np_):
    if kind == "unique":
        bk = rng.permutation(nb).astype(np.int32)
        return bk, rng.integers(0, 2 * nb, size=np_).astype(np.int32)
    if kind == "one_key":
        return np.full(nb, 7, np.int64), rng.integers(6, 9, size=np_).astype(np.int64)
    if kind == "repeated":
        vals = rng.integers(-2**63, 2**63 - 1, size=max(1, nb // 5), dtype=np.int64)
        return vals[rng.integers(0, vals.size, size=nb)], vals[rng.integers(0, vals.size, size=np_)]
    if kind == "all_ones32":  # span 2^32 - 1: one offset from the minimum is carried as all ones
        bk = rng.integers(-2**31, 2**31, size=nb).astype(np.int32)
        bk[:3] = [-2**31, 2**31 - 1, ONES32]
        pk = rng.choice(bk, size=np_)
        pk[::3], pk[::5] = 2**31 - 1, ONES32
        return bk, pk
    if kind == "all_ones64":  # keys that do not narrow
        bk = rng.integers(-2**62, 2**62, size=nb, dtype=np.int64)
        bk[:3] = [-2**63, ONES64, 2**62]
        bk[3::1000] = ONES64
        bk[4::1000] = -1
        pk = rng.choice(bk, size=np_)
        pk[::4], pk[::7], pk[::9] = 2**63 - 1, ONES64, -1
        return bk, pk
    return rng.permutation(nb).astype(np.int64), (rng.integers(0, nb, size=np_) + nb).astype(np.int64)  # none match


@pytest.mark.parametrize("kind", ["unique", "one_key", "repeated", "all_ones32", "all_ones64", "none"])
@pytest.mark.parametrize("nb", [3, 2 * 4608 - 1, 2 * 4608 + 70, 60_001])
@pytest.mark.parametrize("pay", [np.int32, np.int64])
def test_sum_with_carried_payloads(eiger, oracle_mod, kind, nb, pay):
    rng = np.random.default_rng(nb * 31 + len(kind))
    np_ = 37_003 if kind != "one_key" else 2_003
    bk, pk = _keys(kind, rng, nb, np_)
    info = np.iinfo(pay)
    bp = rng.integers(info.min, info.max, size=nb, dtype=np.int64).astype(pay)
    pp = rng.integers(info.min, info.max, size=np_, dtype=np.int64).astype(pay)
    expect = oracle_mod.join_sum(bk, bp, pk, pp)
    t = [torch.from_numpy(a).cuda() for a in (bk, bp, pk, pp)]
    span = int(bk.max()) - int(bk.min())
    for variant, b1, b2 in (("phj1", 1, 0), ("phj2", 3, 4)):
        knobs = eiger.Plan(variant, b1, b2, 1 if bk.dtype == np.int32 or span < 2**32 else 0)
        s, c, used = eiger.join_sum(*t, variant=variant, knobs=knobs, materialize="gftr")
        assert used.materialize == "gftr" and (s, c) == expect, (variant, s, c, expect)
