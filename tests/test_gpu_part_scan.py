"""The scan of the partitioning counts at the edges of its chunks (8192 counts):
a whole number of chunks, one count more and fewer, more chunks than the last
block scans in one round, and a second pass without rows. Every build key is
unique and every probe key drawn from the build (or outside its range), so the
exact result is one pair per matching probe row whose keys are equal."""

import pytest
import torch

pytestmark = pytest.mark.gpu

TILE = 4096  # divides the tile of any build of the kernels


@pytest.fixture(scope="module")
def eiger():
    from paper_2607_04489_gb300 import eiger

    eiger.load()
    return eiger


@pytest.mark.parametrize("bits,np_", [
    ((6, 0), 254 * TILE), ((6, 0), 256 * TILE), ((6, 0), 256 * TILE + 1), ((6, 0), 258 * TILE - 3),
    ((12, 0), 4 * TILE), ((12, 0), 4 * TILE + 1), ((12, 0), 2060 * TILE + 5),  # 515 chunks and more
    ((1, 0), 1), ((1, 1), TILE), ((6, 7), 100 * TILE + 77), ((4, 5), 3_000_001),
])
@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
def test_scan_chunk_edges(eiger, bits, np_, dtype):
    gen = torch.Generator(device="cuda").manual_seed(np_ % 1000)
    nb = 20_000
    bk = (torch.randperm(nb, generator=gen, device="cuda") * 7 - 1000).to(dtype)
    pk = bk[torch.randint(0, nb, (np_,), generator=gen, device="cuda")]
    drop = torch.rand(np_, generator=gen, device="cuda") < 0.1  # outside the build's range
    pk = torch.where(drop, torch.full_like(pk, 10_000_000), pk)
    knobs = eiger.Plan("phj2" if bits[1] else "phj1", bits[0], bits[1], 1)
    r = eiger.join(bk, pk, variant=knobs.variant, knobs=knobs)
    assert (r.plan.bits1, r.plan.bits2) == bits
    p, b = r.probe_idx.long() & 0xFFFFFFFF, r.build_idx.long() & 0xFFFFFFFF
    want = torch.nonzero(~drop).flatten()
    assert r.count == want.numel()
    assert torch.equal(torch.sort(p).values, want)
    assert bool((bk[b] == pk[p]).all())


@pytest.mark.parametrize("bits", [(6, 0), (4, 5)])
def test_no_probe_row_in_range(eiger, bits):
    bk = torch.arange(5000, dtype=torch.int64, device="cuda")
    pk = torch.full((50_000,), 1 << 40, dtype=torch.int64, device="cuda")
    knobs = eiger.Plan("phj2" if bits[1] else "phj1", bits[0], bits[1], 1)
    assert eiger.join(bk, pk, variant=knobs.variant, knobs=knobs).count == 0
