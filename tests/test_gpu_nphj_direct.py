"""The non-partitioned join's direct-addressed table (dense 32-bit keys) against
the oracle: pairs, columns and sums.

Rows around a probe round's 2048 and a build round's 2048, keys at both ends of
the span and just outside it, int32 and narrowed int64 keys at the ends of their
types, spans at and one past the two words per hash slot up to which the table
is direct-addressed, and repeated keys (chains through next[], up to every build
row the same key). Everything is compared exactly after the canonical sort.
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


def _build(kind, dt, nb, rng):
    info = np.iinfo(dt)
    if kind == "low":  # the type's first keys
        return (rng.permutation(nb).astype(np.int64) + info.min).astype(dt)
    if kind == "high":  # the type's last keys
        return (info.max - rng.permutation(nb).astype(np.int64)).astype(dt)
    if kind == "repeats":
        return rng.integers(-nb // 3, nb // 3 + 1, size=nb).astype(dt)
    if kind == "one":
        return np.full(nb, -5, dt)
    slots = 64  # "last": the widest direct-addressed span; "past": one key more
    while slots < 2 * nb:
        slots *= 2
    top = 2 * slots - (1 if kind == "last" else 0)
    k = rng.choice(top, size=nb, replace=False)
    k[0], k[-1] = 0, top
    return (np.unique(np.concatenate([k[k != top], [top]]))[-nb:] if nb < 3 else k).astype(dt)


@pytest.mark.parametrize("dt", [np.int32, np.int64])
@pytest.mark.parametrize("kind", ["low", "high", "repeats", "one", "last", "past"])
@pytest.mark.parametrize("nb,np_", [(1, 1), (2047, 2049), (5000, 70_001)])
def test_direct_addressed_nphj(eiger, oracle_mod, dt, kind, nb, np_):
    if kind == "one":
        np_ = min(np_, 2049)
    rng = np.random.default_rng(nb + len(kind))
    bk = _build(kind, dt, nb, rng)
    info = np.iinfo(dt)
    pk = rng.choice(bk, size=np_)
    out = np.array([max(info.min, int(bk.min()) - 1), min(info.max, int(bk.max()) + 1), info.min, info.max, 0], dt)
    pk[:: max(1, np_ // 40)] = rng.choice(out, size=pk[:: max(1, np_ // 40)].size)
    tb, tp = torch.from_numpy(bk).cuda(), torch.from_numpy(pk).cuda()
    eb, ep, n = oracle_mod.join(bk, pk)
    bc = rng.integers(-2**62, 2**62, size=bk.size)
    pc = rng.integers(-2**62, 2**62, size=np_)
    w = eiger.join_wide(tb, tp, [torch.from_numpy(bc).cuda()], [torch.from_numpy(pc).cuda()], variant="nphj")
    r = eiger.join(tb, tp, variant="nphj")
    span = int(bk.max()) - int(bk.min())
    slots = 64
    while slots < 2 * nb:
        slots *= 2
    direct = 1 if span < 2 * slots else 0
    if nb > 1:  # (one row has no span)
        assert direct == {"last": 1, "past": 0}.get(kind, direct)
    for x in (r, w):
        assert x.plan.direct == direct
        b, p = (t.cpu().numpy().astype(np.int64) & 0xFFFFFFFF for t in (x.build_idx, x.probe_idx))
        o = np.lexsort((b, p))
        assert x.count == n and x.plan.variant == "nphj"
        np.testing.assert_array_equal(p[o], ep)
        np.testing.assert_array_equal(b[o], eb)
    np.testing.assert_array_equal(w.build_cols[0].cpu().numpy(), bc[b])
    np.testing.assert_array_equal(w.probe_cols[0].cpu().numpy(), pc[p])
    s, c, plan = eiger.join_sum(tb, torch.from_numpy(bc).cuda(), tp, torch.from_numpy(pc).cuda(), variant="nphj")
    assert plan.direct == direct and (s, c) == oracle_mod.join_sum(bk, bc, pk, pc)


def test_workspace_of_the_hash_table_alone(eiger, oracle_mod):
    """4 bytes per build row less than the query says, all that the hash table
    needs: the join runs; one page less: refused."""
    rng = np.random.default_rng(5)
    nb = 100_000
    bk, pk = rng.permutation(nb).astype(np.int32), rng.integers(-10, nb + 10, size=nb).astype(np.int32)
    _, _, n = oracle_mod.join(bk, pk)
    tb, tp = torch.from_numpy(bk).cuda(), torch.from_numpy(pk).cuda()
    query = eiger.join_workspace(nb, nb, eiger.I32, "nphj")
    ob, op = (torch.empty(nb, dtype=torch.int32, device="cuda") for _ in range(2))
    for less, status in ((0, eiger.OK), (4 * nb, eiger.OK), (4 * nb + 4096, eiger.ERR_WORKSPACE)):
        ws = torch.empty(query - less, dtype=torch.uint8, device="cuda")
        st, cnt, plan = eiger.join_into(tb, tp, variant="nphj", out_bidx=ob, out_pidx=op, capacity=nb, workspace=ws)
        assert st == status
        if st == eiger.OK:
            assert plan.direct == (1 if less == 0 else 0)
            assert cnt == n and bool((tb[ob[:n].long()] == tp[op[:n].long()]).all())
            assert torch.unique(op[:n]).numel() == n
