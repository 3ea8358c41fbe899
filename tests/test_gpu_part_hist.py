"""The digit counts of the partitioning passes: a CTA per tile (inputs of few
tiles), a warp per tile (many), key columns that start off a 16-byte boundary,
tiles of a few rows, and rows outside the build's range. Every build key is
unique and every probe key drawn from the build, so the exact result is one pair
per kept probe row whose keys are equal."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eiger():
    from paper_2607_04489_gb300 import eiger

    eiger.load()
    return eiger


@pytest.mark.parametrize("np_", [1, 3, 5, 511, 513, 4095, 4097, 300_001, 45_000_003])  # the last: a warp per tile
@pytest.mark.parametrize("lead", [0, 1, 3])  # rows cut off the front of the columns
@pytest.mark.parametrize("dtype,narrow", [(torch.int32, 1), (torch.int64, 1), (torch.int64, 0)])
def test_hist_tiles_and_alignment(eiger, np_, lead, dtype, narrow):
    gen = torch.Generator(device="cuda").manual_seed(np_ % 997 + lead)
    nb = 30_000
    bk = torch.randperm(nb + lead, generator=gen, device="cuda").to(dtype) * 5 - 77
    pk = bk[lead:][torch.randint(0, nb, (np_ + lead,), generator=gen, device="cuda")]
    pk[lead::7] = 40_000_000  # outside the build's range
    bk, pk = bk[lead:], pk[lead:]
    if not narrow:  # spread over 64 bits: odd multiplier, wraps
        bk, pk = bk * 6364136223846793005, pk * 6364136223846793005
    knobs = eiger.Plan("phj2", 4, 5, narrow)
    r = eiger.join(bk, pk, variant="phj2", knobs=knobs)
    assert r.plan.narrow == narrow
    keep = torch.ones(np_, dtype=torch.bool, device="cuda")
    keep[0::7] = False
    want = torch.nonzero(keep).flatten()
    p, b = r.probe_idx.long() & 0xFFFFFFFF, r.build_idx.long() & 0xFFFFFFFF
    assert r.count == want.numel()
    assert torch.equal(torch.sort(p).values, want)
    assert bool((bk[b] == pk[p]).all())
