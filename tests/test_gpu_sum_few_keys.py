"""The carried sum with far more build rows than keys: a partition's build rows go
to direct-addressed tables in chunks of at most 131,072 rows, whose sums add up.
Build sides on each side of one chunk, of one and of a few keys, exactly against
closed forms; and the time of a build column of two keys against a dense one's,
so that one CTA does not take all rows of a key."""

import pytest
import torch

pytestmark = pytest.mark.gpu

CHUNK = 131_072


@pytest.fixture(scope="module")
def eiger():
    from paper_2607_04489_gb300 import eiger

    eiger.load()
    return eiger


def _mod64(x):
    return (x + (1 << 63)) % (1 << 64) - (1 << 63)


@pytest.mark.parametrize("nb", [CHUNK - 1, CHUNK, CHUNK + 1, 5 * CHUNK + 77])
@pytest.mark.parametrize("keys", [1, 3])
@pytest.mark.parametrize("pay", [torch.int32, torch.int64])
def test_few_keys(eiger, nb, keys, pay):
    gen = torch.Generator(device="cuda").manual_seed(nb + keys)
    big = (1 << 30) if pay == torch.int32 else (1 << 62)
    bk = torch.randint(0, keys, (nb,), generator=gen, device="cuda", dtype=torch.int32)
    pk = torch.randint(0, keys + 1, (70_001,), generator=gen, device="cuda", dtype=torch.int32)  # some absent
    bp = torch.randint(-big, big, (nb,), generator=gen, device="cuda", dtype=pay)
    pp = torch.randint(-big, big, (pk.numel(),), generator=gen, device="cuda", dtype=pay)
    total = count = 0
    for k in range(keys):
        mb, mp = bk == k, pk == k
        rb, rp = int(mb.sum()), int(mp.sum())
        total += rp * int(bp[mb].long().sum()) + rb * int(pp[mp].long().sum())
        count += rb * rp
    knobs = eiger.Plan("phj1", 1, 0, 1)
    s, c, plan = eiger.join_sum(bk, bp, pk, pp, variant="phj1", knobs=knobs, materialize="gftr")
    assert (s, c, plan.direct) == (_mod64(total), count, 1)


def test_few_keys_spread_over_the_chip(eiger):
    """Two keys on 2^24 build rows take at most 20 times a dense column's time in
    the sum's kernel (one CTA per key: 66 times)."""
    nb = 1 << 24
    dense = torch.randperm(nb, device="cuda").to(torch.int32)
    pay = torch.ones(nb, dtype=torch.int32, device="cuda")

    def ms(bk, pk, bits):
        best = float("inf")
        for _ in range(4):
            _, c, _ = eiger.join_sum(bk, pay, pk, pay[:pk.numel()], variant="phj2",
                                     knobs=eiger.Plan("phj2", bits, bits, 1), materialize="gftr")
            assert c == pk.numel() * (nb // int(bk.max() + 1))
            best = min(best, sum(m for name, m, _, _ in eiger.profile_read() if name == "phj_sum"))
        return best

    eiger.profile(True)
    try:
        assert ms(dense % 2, dense[:1000] % 2, 1) < 20 * ms(dense, dense, 6)
    finally:
        eiger.profile(False)
