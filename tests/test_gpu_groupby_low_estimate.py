"""Group-bys whose sketch sees far fewer groups than there are.

The sketch hashes keys with a bijection, so keys can be chosen by their hash:
every register of rank 1 makes the estimate about 23,600 whatever the number of
keys, a few registers only make it a few hundred. The first plan's tables then
overflow; the retries must reach the exact result, as quickly as the largest
tables allow.
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


def _unhash(h):
    """Inverse of the SplitMix64 output function on uint64 arrays."""
    u = np.uint64
    inv = lambda a: u(pow(a, -1, 1 << 64))
    h = h ^ (h >> u(31)) ^ (h >> u(62))
    h = h * inv(0x94D049BB133111EB)
    h = h ^ (h >> u(27)) ^ (h >> u(54))
    h = h * inv(0xBF58476D1CE4E5B9)
    return h ^ (h >> u(30)) ^ (h >> u(60))


def _keys(groups, registers, rng):
    """Distinct int64 keys in the first `registers` registers, all of rank 1."""
    low = rng.permutation(1 << 22)[:groups].astype(np.uint64) * np.uint64(0x1234567) + (np.uint64(1) << np.uint64(49))
    reg = rng.integers(0, registers, size=groups).astype(np.uint64)
    return _unhash((reg << np.uint64(50)) | low).astype(np.int64)


@pytest.mark.parametrize("registers,estimate", [(1 << 14, 23_600), (256, 260)])
@pytest.mark.parametrize("variant", ["auto", "hash", "partition"])
def test_low_estimate(eiger, oracle_mod, registers, estimate, variant):
    rng = np.random.default_rng(registers)
    groups = 1 << 20
    vals = _keys(groups, registers, rng)
    assert np.unique(vals).size == groups
    keys = np.concatenate([vals, vals[rng.integers(0, groups, size=groups // 2)]])
    rng.shuffle(keys)
    v = rng.integers(-2**31, 2**31, size=keys.size).astype(np.int32)
    ok, oa = oracle_mod.groupby(keys, [("sum", v), ("count", None)])
    r = eiger.groupby(torch.from_numpy(keys).cuda(), [("sum", torch.from_numpy(v).cuda()), ("count", None)],
                      variant=variant, capacity=groups)
    assert abs(r.plan.estimate / estimate - 1) < 0.05
    assert r.groups == groups
    gk = r.keys.cpu().numpy()
    order = np.argsort(gk)
    np.testing.assert_array_equal(gk[order], ok)
    for got, want in zip(r.aggs, oa):
        np.testing.assert_array_equal(got.cpu().numpy()[order], want)
    if variant == "partition":
        # with tables of 4096 slots from the second attempt on: the fewest bits
        # in steps of 2 from the first plan's that leave fewer groups a partition
        bits = max(1, int(np.ceil(np.log2(r.plan.estimate / 1024))))
        attempts = 1
        while groups / 2**bits > 3500:
            bits += 2
            attempts += 1
        assert r.plan.attempts == attempts and r.plan.bits1 + r.plan.bits2 == bits
