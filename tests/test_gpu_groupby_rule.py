"""The group-by AUTO takes: shared-memory tables for few groups; beyond them the
global table below 2^24 rows, and for keys without aggregates at any size; else the
partitions. Groups and sums against torch."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eiger():
    from paper_2607_04489_gb300 import eiger

    eiger.load()
    return eiger


@pytest.mark.parametrize("rows,groups,aggs,variant", [
    (1 << 24, 1000, 1, "hash"),
    (1 << 24, 40_000, 0, "hash"),
    (1 << 24, 40_000, 1, "partition"),
    ((1 << 24) - 1, 40_000, 1, "hash"),
    (1 << 24, 1 << 23, 0, "partition"),  # the global table leaves half of L2
])
@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
def test_auto_variant(eiger, rows, groups, aggs, variant, dtype):
    gen = torch.Generator(device="cuda").manual_seed(groups)
    ids = torch.randint(0, groups, (rows,), generator=gen, device="cuda")
    keys = ids.to(torch.int32) * 3 if dtype == torch.int32 else ids * 4_000_000_007
    vals = torch.randint(-2**31, 2**31, (rows,), generator=gen, device="cuda").to(torch.int32)
    want = torch.unique(keys)
    r = eiger.groupby(keys, [("sum", vals)] * aggs, capacity=groups)
    assert r.plan.variant == variant and r.groups == want.numel()
    got, order = torch.sort(r.keys)
    assert torch.equal(got, want)
    if aggs:
        sums = torch.zeros(groups, dtype=torch.int64, device="cuda").scatter_add_(0, ids, vals.long())
        assert torch.equal(r.aggs[0][order], sums[torch.unique(ids)])
