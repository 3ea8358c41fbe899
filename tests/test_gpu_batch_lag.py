"""The staged order of a batch's items: a join's clear, build and probe items
lie `lag` stages apart, from 1 (large tables) to 128 (small joins), which may be
more stages than there are joins. Exact pairs per join against the oracle, for
batches on each side of those limits; int32 and int64 keys, and load factors
whose slot counts sit beside a power of two."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eiger():
    from paper_2607_04489_gb300 import eiger

    eiger.load()
    return eiger


# (build rows per join, probe rows per join, joins checked against the oracle)
BATCHES = {
    "one_join": ([9000], [20_000], [0]),
    "three_joins_one_empty": ([5000, 0, 5000], [5000, 4000, 1], [0, 1, 2]),
    "more_than_the_largest_lag": ([64 + j % 200 for j in range(700)], [1 + j % 150 for j in range(700)],
                                  list(range(0, 700, 37)) + [699]),
    "tables_bound_the_lag": ([3_000_000, 10, 2_000_000], [50_000, 50_000, 50_000], [0, 1, 2]),
    "slots_at_a_power_of_two": ([57, 58, 115, 116, 3686, 3687], [500] * 6, list(range(6))),
}


@pytest.mark.parametrize("dtype", [np.int32, np.int64])
@pytest.mark.parametrize("load", [0.5, 0.9])
@pytest.mark.parametrize("case", sorted(BATCHES))
def test_batch_stages(eiger, oracle_mod, case, load, dtype):
    nbs, nps, check = BATCHES[case]
    rng = np.random.default_rng(len(nbs))
    builds, probes = [], []
    for nb, n in zip(nbs, nps):
        bk = (rng.permutation(2 * nb)[:nb] - 50).astype(dtype)  # half the range, no key twice
        builds.append(bk)
        probes.append(rng.integers(-60, 2 * nb + 1, size=n).astype(dtype))
    bj = eiger.BatchedJoin([torch.from_numpy(b).cuda() for b in builds], [torch.from_numpy(p).cuda() for p in probes],
                           knobs=eiger.BatchKnobs(512, 4096, load))
    bj.run()
    torch.cuda.synchronize()
    assert int(bj.status) == 0
    for j in check:
        n, gb, gp = bj.result(j)
        eb, ep, en = oracle_mod.join(builds[j], probes[j])
        assert n == en
        b, p = gb.cpu().numpy().astype(np.int64) & 0xFFFFFFFF, gp.cpu().numpy().astype(np.int64) & 0xFFFFFFFF
        o = np.lexsort((b, p))
        np.testing.assert_array_equal(b[o], eb.astype(np.int64))
        np.testing.assert_array_equal(p[o], ep.astype(np.int64))
