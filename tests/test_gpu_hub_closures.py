"""Frontier closures of relations in which nearly every row is one fact to a hub: the rows that follow from the hub's are
expanded after all when their levels are not certain, by the whole GPU."""
import time

import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pkg = pytest.importorskip("paper_2408_10369_gb300")
from paper_2408_10369_gb300 import bmlp  # noqa: E402

pytestmark = pytest.mark.gpu
PACKED = bmlp.BMLP_FMT_PACKED64


def relation(kind, n):
    k = np.arange(1, n)
    if kind == "star":  # all constants and the hub have facts with one another
        return wl.csr_from_pairs(n, np.concatenate([k, 0 * k]), np.concatenate([0 * k, k]))
    m = n // 10         # constants by way of n / 10 others to the hub, and the hub to all
    mid = 1 + k % m
    return wl.csr_from_pairs(n, np.concatenate([k, 0 * k]), np.concatenate([np.where(k <= m, 0, mid), k]))


@pytest.mark.parametrize("kind,n", [("star", 4200), ("star", 9001), ("star", 30000), ("spokes", 5000), ("spokes", 12000)])
def test_hub_closures(kind, n):
    csr = relation(kind, n)
    R = torch.from_numpy(wl.csr_to_packed(n, *csr).view(np.int64)).cuda()
    out = torch.zeros_like(R)
    rows = np.arange(n, dtype=np.int32) if n < 10000 else np.unique(np.linspace(0, n - 1, 300).astype(np.int32))
    want, depth, _ = oracle.reach_rows(n, *csr, rows)
    with pkg.Context(0) as ctx:
        best = 1e9
        for _ in range(5):
            torch.cuda.synchronize()
            t = time.perf_counter()
            it = ctx.rms(R, n, out, fmt=PACKED, variant="smp_packed")
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
            assert it >= int(depth.max()) + 1 and (n >= 10000 or it == int(depth.max()) + 1)
        assert ctx.stats()["sliced_closures"] == 1
    np.testing.assert_array_equal(wl.unpack_rows(out.cpu().numpy().view(np.uint64)[rows], n), want)
    assert best < 1e-3 + n * n * 15e-12  # one CTA for those rows: n * n * 120e-12
