"""Calls of several host threads at once whose kernels take different amounts of
shared memory: the same kernel, with tables of 64 KB in one thread and of a few
hundred bytes in another. Every call must succeed with the exact result."""

import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eiger():
    from paper_2607_04489_gb300 import eiger

    eiger.load()
    return eiger


def _run(workers):
    errors = []

    def body(make, calls):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                call = make()
                for _ in range(calls):
                    call()
        except Exception as e:  # noqa: BLE001 (reported by the test)
            errors.append(repr(e))

    threads = [threading.Thread(target=body, args=w) for w in workers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]


def test_joins_with_tables_of_different_sizes(eiger):
    nb = 1 << 15
    bk = torch.from_numpy(np.random.default_rng(0).permutation(nb).astype(np.int32)).cuda()
    pk = bk[: nb // 2].contiguous()
    torch.cuda.synchronize()

    def join(bits):
        def make():
            knobs = eiger.Plan("phj1", bits, 0, 1)
            ws = torch.empty(eiger.join_workspace(nb, nb // 2, eiger.I32, "phj1", knobs), dtype=torch.uint8, device="cuda")
            ob, op = (torch.empty(nb // 2, dtype=torch.int32, device="cuda") for _ in range(2))

            def call():
                st, n, _ = eiger.join_into(bk, pk, variant="phj1", knobs=knobs, out_bidx=ob, out_pidx=op,
                                           capacity=nb // 2, workspace=ws)
                if st != eiger.OK:
                    raise RuntimeError(eiger.last_error())
                assert n == nb // 2

            return call

        return make

    _run([(join(b), 1500) for b in (1, 8, 1, 8)])  # 2^14 and 2^7 slots


def test_groupbys_with_tables_of_different_sizes(eiger):
    key = torch.from_numpy(np.random.default_rng(1).integers(0, 3000, 30_000).astype(np.int32)).cuda()
    torch.cuda.synchronize()

    def groupby(bits):
        def make():
            knobs = eiger.GbPlan("partition", bits1=bits, bits2=0)
            aggs = [("sum", key), ("max", key), ("min", key), ("count", None)]
            ws = torch.empty(eiger.groupby_workspace(key.numel(), eiger.I32, aggs, "partition"), dtype=torch.uint8,
                             device="cuda")
            ok = torch.empty(3000, dtype=torch.int32, device="cuda")
            outs = [torch.empty(3000, dtype=torch.int64, device="cuda") for _ in aggs]

            def call():
                st, n, _ = eiger.groupby_into(key, aggs, ok, outs, variant="partition", knobs=knobs, capacity=3000,
                                              workspace=ws)
                if st != eiger.OK:
                    raise RuntimeError(eiger.last_error())
                assert n == 3000

            return call

        return make

    _run([(groupby(b), 1500) for b in (2, 9, 2, 9)])
