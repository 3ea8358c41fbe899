"""Repeated build keys in the partitioned join's direct-addressed tables.

An item whose keys repeat goes to a launch whose tables chain up to 1024 further
rows; one with more goes to another in pieces of at most 4096 build rows. The
cases lie on each side of both limits, against the oracle in every output mode,
and the time of a column with a few repeats is held against the unique column's.
"""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

CHAINS = 1024  # further rows a table holds


@pytest.fixture(scope="module")
def eiger():
    from paper_2607_04489_gb300 import eiger

    eiger.load()
    return eiger


def _canon(b, p, *cols):
    b, p = (np.asarray(x.cpu()).astype(np.int64) & 0xFFFFFFFF for x in (b, p))
    o = np.lexsort((b, p))
    return (b[o], p[o], *[c.cpu().numpy()[o] for c in cols])


SPAN = 1 << 18


def _build(kind, rng):
    """Dense keys [0, SPAN) and, over them, the repeats of `kind`; few enough in
    all that the join still takes direct-addressed tables (97 % distinct)."""
    base = rng.permutation(SPAN)
    if kind == "pairs":  # keys twice: chains of one entry
        more = rng.choice(SPAN, 3000, replace=False)
    elif kind == "one_chain":  # one key, as often as one table's chains hold beside a full table
        more = np.full(CHAINS, 77)
    elif kind == "one_too_many":  # of a full table
        more = np.full(CHAINS + 1, 77)
    elif kind == "one_too_many_sparse":  # found only when the chains are full
        base = base[base % 10 != 3]
        more = np.full(CHAINS + 1, 77)
    elif kind == "mixed":  # chains of different lengths, some keys many times, in every partition
        more = np.concatenate([np.repeat(rng.choice(SPAN, 60, replace=False), np.arange(60)), rng.choice(SPAN, 1000)])
    else:  # "default": one key on many rows, several pieces; others repeated beside it
        more = np.concatenate([np.full(4_000, 12_345), rng.choice(SPAN, 200)])
    return rng.permutation(np.concatenate([base, more]))


@pytest.mark.parametrize("kind", ["pairs", "one_chain", "one_too_many", "one_too_many_sparse", "mixed", "default"])
@pytest.mark.parametrize("bits", [(4, 0), (4, 1), (5, 4)])  # 2^14, 2^13 and 2^9 slots
@pytest.mark.parametrize("dtype", [np.int32, np.int64])
def test_repeats_in_direct_tables(eiger, oracle_mod, kind, bits, dtype):
    rng = np.random.default_rng(len(kind) + sum(bits))
    bk = (_build(kind, rng) - 5_000).astype(dtype)
    pk = rng.integers(-6_000, SPAN - 4_000, size=70_003).astype(dtype)
    pk[:300] = bk[:300]
    rows = np.bincount(bk + 5_000, minlength=SPAN)[np.clip(pk + 5_000, 0, SPAN - 1)]
    pk[(rows > 500) & (rng.random(pk.size) < 0.5)] = -5_999
    pk[1000:1003] = 12_345 - 5_000
    variant = "phj2" if bits[1] else "phj1"
    knobs = eiger.Plan(variant, bits[0], bits[1], 1)
    tb, tp = torch.from_numpy(bk).cuda(), torch.from_numpy(pk).cuda()
    eb, ep, n = oracle_mod.join(bk, pk)

    r = eiger.join(tb, tp, variant=variant, knobs=knobs)
    b, p = _canon(r.build_idx, r.probe_idx)
    assert r.count == n and r.plan.direct == 1
    np.testing.assert_array_equal(p, ep)
    np.testing.assert_array_equal(b, eb)

    bc = rng.integers(-2**62, 2**62, size=bk.size)
    pc = rng.integers(-2**62, 2**62, size=pk.size)
    cb, cp = torch.from_numpy(bc).cuda(), torch.from_numpy(pc).cuda()
    for mat in ("gftr", "gfur"):
        w = eiger.join_wide(tb, tp, [cb], [cp], variant=variant, knobs=knobs, materialize=mat)
        b, p, b0, p0 = _canon(w.build_idx, w.probe_idx, *w.build_cols, *w.probe_cols)
        assert w.count == n
        np.testing.assert_array_equal(p, ep)
        np.testing.assert_array_equal(b, eb)
        np.testing.assert_array_equal(b0, bc[b])
        np.testing.assert_array_equal(p0, pc[p])
        s, c, _ = eiger.join_sum(tb, cb, tp, cp, variant=variant, knobs=knobs, materialize=mat)
        assert (s, c) == oracle_mod.join_sum(bk, bc, pk, pc)


def _join_ms(eiger, bk, pk, cols):
    """Fastest of five runs of the join stages of a dense partitioned join."""
    knobs = eiger.Plan("phj2", 5, 5, 1)
    cap = pk.numel() + pk.numel() // 4
    best = float("inf")
    eiger.profile(True)
    try:
        for _ in range(5):
            if cols:
                eiger.join_wide(bk, pk, [bk], [pk], indices=False, variant="phj2", knobs=knobs, materialize="gftr",
                                capacity=cap)
            else:
                eiger.join(bk, pk, variant="phj2", knobs=knobs, capacity=cap)
            best = min(best, sum(ms for name, ms, _, _ in eiger.profile_read() if name.startswith("phj_join")))
    finally:
        eiger.profile(False)
    return best


@pytest.mark.parametrize("cols", [False, True])
def test_few_repeats_cost_little(eiger, cols):
    """1 % repeated rows, in every partition: the join's kernels take no more
    than 2.5 times what they take on unique keys."""
    nb, np_ = 1 << 23, 1 << 25
    gen = torch.Generator(device="cuda").manual_seed(1)
    bk = torch.randperm(nb, generator=gen, device="cuda").to(torch.int32)
    pk = torch.randint(0, nb, (np_,), generator=gen, device="cuda").to(torch.int32)
    rep = bk.clone()
    rep[: nb // 100] = rep[nb // 2: nb // 2 + nb // 100]
    assert _join_ms(eiger, rep, pk, cols) < 2.5 * _join_ms(eiger, bk, pk, cols)


@pytest.mark.parametrize("cols", [False, True])
def test_default_key_costs_little(eiger, cols):
    """One key on 2 % of the build rows that no probe row asks for: the join's
    kernels take no more than 4 times what they take on unique keys (its rows on one
    CTA, or in hash tables whose equal keys the probes walk: tens)."""
    nb, np_ = 1 << 23, 1 << 25
    gen = torch.Generator(device="cuda").manual_seed(2)
    bk = torch.randperm(nb, generator=gen, device="cuda").to(torch.int32)
    pk = torch.randint(0, nb, (np_,), generator=gen, device="cuda").to(torch.int32)
    pk += (pk == 777).to(torch.int32)
    rep = bk.clone()
    rep[: nb // 50] = 777
    assert _join_ms(eiger, rep, pk, cols) < 4 * _join_ms(eiger, bk, pk, cols)
