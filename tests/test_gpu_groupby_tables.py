"""The group-by's shared-memory tables (CTA tables of the hash variant, one
table per partition of the partition variant) against the oracle.

Aggregates are held in 32-bit words where the type allows, so the cases drive
the carry between a sum's halves (mixed signs, values next to +-2^31 and 2^63,
sums that wrap modulo 2^64), MIN and MAX at the types' limits, and every count
of aggregates with 4- and 8-byte columns. Group counts run from one (a copy of
the aggregates per lane) over the largest a CTA table takes to past it, and
partitions are cut into several items (few groups) or taken whole. All results
are integers: compared exactly.
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


def _values(rng, n, dt, kind):
    info = np.iinfo(dt)
    if kind == "limits":  # around the ends of the type and zero
        return rng.choice(np.array([info.min, info.min + 1, -1, 0, 1, info.max - 1, info.max], dt), size=n)
    return rng.integers(info.min, info.max, size=n, dtype=np.int64).astype(dt)


AGGS = {
    "sum32": [("sum", np.int32)],
    "max64": [("max", np.int64)],
    "sum32_max32": [("sum", np.int32), ("max", np.int32)],
    "count_sum64": [("count", None), ("sum", np.int64)],
    "min32_sum32_count": [("min", np.int32), ("sum", np.int32), ("count", None)],
    "all": [("sum", np.int64), ("min", np.int64), ("max", np.int32), ("sum", np.int32)],
}


@pytest.mark.parametrize("aggs", sorted(AGGS))
@pytest.mark.parametrize("groups", [1, 31, 700, 3500, 9000, 14000])
@pytest.mark.parametrize("variant", ["hash", "partition"])
def test_groupby_shared_memory_tables(eiger, oracle_mod, aggs, groups, variant):
    rng = np.random.default_rng(groups * 7 + len(aggs))
    n = 150_013
    wide = groups % 2 == 1  # odd counts: keys that do not narrow
    vals = (rng.permutation(groups).astype(np.int64) * (1_000_000_007 if wide else 3) - 1_000).astype(
        np.int64 if wide else np.int32)
    keys = vals[rng.integers(0, groups, size=n)]
    keys[rng.integers(0, n, size=n // 3)] = vals[0]  # a hot group
    cols = [(op, None if dt is None else _values(rng, n, dt, "limits" if q % 2 else "uniform"))
            for q, (op, dt) in enumerate(AGGS[aggs])]
    ok, oa = oracle_mod.groupby(keys, cols)
    r = eiger.groupby(torch.from_numpy(keys).cuda(),
                      [(op, None if v is None else torch.from_numpy(v).cuda()) for op, v in cols], variant=variant)
    assert r.groups == ok.size and r.plan.variant == variant
    gk = r.keys.cpu().numpy().astype(np.int64)
    order = np.argsort(gk)
    np.testing.assert_array_equal(gk[order], ok)
    for got, want in zip(r.aggs, oa):
        np.testing.assert_array_equal(got.cpu().numpy()[order], want)
