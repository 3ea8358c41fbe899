"""The partitioned join's direct-addressed tables (dense, hardly repeated 32-bit
build keys) against the oracle, in every output mode.

Plans put the slots of a partition above the largest table (hash tables then), at
it, one bit below it and at a handful; a span one past a power of two and an
eighth-full span set the density limits. A few repeated build keys send their
partitions (larger than one hash table) through the later launches beside
partitions that stay in the first, and a hot probe key cuts its partition's probe
side into several items. plan_used says which tables ran. Pairs and columns are
compared after the canonical sort, sums exactly.
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


def _input(kind, rng):
    nb, np_ = 40_000, 150_000
    if kind == "dense":  # one past a power of two would double the span: 2^15 + 1 .. 2^16 slots
        bk = rng.permutation(nb).astype(np.int64) + 10**12
    elif kind == "sparse":  # an eighth of 2^18 slots, and the span's last key
        nb = 1 << 15
        bk = np.append(rng.choice((1 << 18) - 1, size=nb - 2, replace=False) + 0, [0, (1 << 18) - 1]).astype(np.int32)
        bk = np.unique(bk)
        extra = np.setdiff1d(np.arange(1 << 18, dtype=np.int32), bk)[: nb - bk.size]
        bk = rng.permutation(np.concatenate([bk, extra])).astype(np.int32)
    elif kind == "repeats":  # a few keys twice or more: their partitions leave direct addressing
        bk = rng.permutation(nb).astype(np.int32) - 20_000
        bk[:40] = bk[100]
        bk[50:60] = bk[200:210]
    else:  # tiny
        bk, np_ = np.array([5, 3, 4, 9], np.int32), 1000
    pk = rng.choice(bk, size=np_)
    pk[: np_ // 2] = bk[min(100, bk.size - 1)]  # a hot key: more probe rows than one item takes
    if kind == "repeats":
        pk = pk[np_ // 2 - 2_000:]
    miss = rng.random(pk.size) < 0.1
    pk = np.where(miss, pk + int(bk.max()) - int(bk.min()) + 1, pk).astype(bk.dtype)
    return bk, pk


def _canon(b, p, *cols):
    b, p = (np.asarray(x.cpu()).astype(np.int64) & 0xFFFFFFFF for x in (b, p))
    o = np.lexsort((b, p))
    return (b[o], p[o], *[c.cpu().numpy()[o] for c in cols])


@pytest.mark.parametrize("kind", ["dense", "sparse", "repeats", "tiny"])
@pytest.mark.parametrize("bits", [(2, 0), (2, 1), (4, 0), (5, 6)])
def test_direct_addressed_joins(eiger, oracle_mod, kind, bits):
    rng = np.random.default_rng(len(kind) + 10 * sum(bits))
    bk, pk = _input(kind, rng)
    variant = "phj2" if bits[1] else "phj1"
    knobs = eiger.Plan(variant, bits[0], bits[1], 1)
    tb, tp = torch.from_numpy(bk).cuda(), torch.from_numpy(pk).cuda()
    eb, ep, n = oracle_mod.join(bk, pk)

    kbits = max(2, (int(bk.max()) - int(bk.min())).bit_length())
    direct = 1 if kbits - sum(bits) <= 14 else 0  # slots; at most 2^13 for the carried sum

    r = eiger.join(tb, tp, variant=variant, knobs=knobs)
    b, p = _canon(r.build_idx, r.probe_idx)
    assert r.count == n and r.plan.direct == direct
    np.testing.assert_array_equal(p, ep)
    np.testing.assert_array_equal(b, eb)

    bcols = [rng.integers(-2**31, 2**31, size=bk.size).astype(np.int32), rng.integers(-2**62, 2**62, size=bk.size)]
    pcols = [rng.integers(-2**62, 2**62, size=pk.size), rng.integers(-2**31, 2**31, size=pk.size).astype(np.int32)]
    for mat in ("gftr", "gfur"):
        w = eiger.join_wide(tb, tp, [torch.from_numpy(c).cuda() for c in bcols],
                            [torch.from_numpy(c).cuda() for c in pcols], variant=variant, knobs=knobs, materialize=mat)
        b, p, b0, b1, p0, p1 = _canon(w.build_idx, w.probe_idx, *w.build_cols, *w.probe_cols)
        assert w.count == n and w.plan.materialize == mat and w.plan.direct == direct
        np.testing.assert_array_equal(p, ep)
        np.testing.assert_array_equal(b, eb)
        for got, want in ((b0, bcols[0][b]), (b1, bcols[1][b]), (p0, pcols[0][p]), (p1, pcols[1][p])):
            np.testing.assert_array_equal(got, want)
        s, c, plan = eiger.join_sum(tb, torch.from_numpy(bcols[1]).cuda(), tp, torch.from_numpy(pcols[0]).cuda(),
                                    variant=variant, knobs=knobs, materialize=mat)
        assert plan.direct == (direct if mat == "gfur" else 1 if kbits - sum(bits) <= 13 else 0)
        assert (s, c) == oracle_mod.join_sum(bk, bcols[1], pk, pcols[0])


def test_direct_addressed_join_capacity(eiger, oracle_mod):
    """Exactly the count, and one entry less: nothing past the capacity."""
    rng = np.random.default_rng(3)
    bk, pk = _input("repeats", rng)
    tb, tp = torch.from_numpy(bk).cuda(), torch.from_numpy(pk).cuda()
    knobs = eiger.Plan("phj1", 2, 0, 1)
    _, _, n = oracle_mod.join(bk, pk)
    ws = torch.empty(eiger.join_workspace(bk.size, pk.size, eiger.I32, "phj1", knobs), dtype=torch.uint8, device="cuda")
    for cap in (n, n - 1):
        ob, op = (torch.full((n + 64,), -7, dtype=torch.int32, device="cuda") for _ in range(2))
        st, cnt, _ = eiger.join_into(tb, tp, variant="phj1", knobs=knobs, out_bidx=ob, out_pidx=op, capacity=cap,
                                     workspace=ws)
        assert cnt == n and st == (eiger.OK if cap == n else eiger.ERR_CAPACITY)
        assert bool((ob[cap:] == -7).all()) and bool((op[cap:] == -7).all())


@pytest.mark.parametrize("span_bits,direct", [(18, 1), (19, 0)])
@pytest.mark.parametrize("mode", ["pairs", "columns", "gfur", "gftr"])
def test_density_limit(eiger, span_bits, direct, mode):
    """2^15 build rows: direct-addressed over a span of an eighth's density, 2^18
    keys, and no more over one key further (2^18 + 1, which counts as 2^19)."""
    rng = np.random.default_rng(span_bits)
    nb, top = 1 << 15, (1 << 18) - (1 if span_bits == 18 else 0)
    bk = np.append(rng.choice(np.arange(1, top), size=nb - 2, replace=False), [0, top]).astype(np.int32)
    tb = torch.from_numpy(bk).cuda()
    pay = torch.ones(nb, dtype=torch.int32, device="cuda")
    bits = 6 if mode == "gftr" else 5
    knobs = eiger.Plan("phj1", bits, 0, 1)
    if mode == "pairs":
        r = eiger.join(tb, tb, variant="phj1", knobs=knobs)
    elif mode == "columns":
        r = eiger.join_wide(tb, tb, [pay], [pay], variant="phj1", knobs=knobs)
    else:
        s, c, plan = eiger.join_sum(tb, pay, tb, pay, variant="phj1", knobs=knobs, materialize=mode)
        assert (s, c, plan.direct) == (2 * nb, nb, direct)
        return
    assert r.count == nb and r.plan.direct == direct
    assert bool((r.build_idx == r.probe_idx).all())


def test_auto_takes_the_dense_plans(eiger):
    """AUTO on dense keys: NPHJ while the table stays in L2, partitions of up to
    2^14 slots (2^13 for carried sums) beyond; on as many sparse keys neither."""
    gen = torch.Generator(device="cuda").manual_seed(1)
    for log2nb, variant in ((23, "nphj"), (26, "phj2")):
        nb = 1 << log2nb
        bk = torch.randperm(nb, generator=gen, device="cuda").to(torch.int32)
        pk = bk[:nb // 2].contiguous()
        r = eiger.join(bk, pk)
        assert r.count == pk.numel() and (r.plan.variant, r.plan.direct) == (variant, 1)
        if variant == "phj2":
            assert r.plan.bits1 + r.plan.bits2 == log2nb - 14
            s = eiger.join_sum(bk, bk, pk, pk, materialize="gftr")[2]
            assert (s.variant, s.direct, s.bits1 + s.bits2) == ("phj2", 1, log2nb - 13)
        del r
        sparse = (bk * 31).contiguous() if log2nb == 26 else (bk * 400).contiguous()
        r = eiger.join(sparse, sparse[:1000].contiguous())
        assert r.count == 1000 and (r.plan.variant, r.plan.direct) == ("phj2", 0)
        del r
