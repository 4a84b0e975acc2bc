"""Insertions of a few facts: up to n = 8,192 three go by one launch each, which take no workspace; four are one chunk, and
above that three are."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pkg = pytest.importorskip("paper_2408_10369_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt", [pkg.BMLP_FMT_PACKED64, pkg.BMLP_FMT_U8])
@pytest.mark.parametrize("n,m", [(1, 3), (65, 3), (700, 3), (700, 4), (2500, 3), (8192, 3), (8193, 3), (8193, 2)])
def test_insertions(n, m, fmt):
    ip, ix = wl.er_graph(n, 0.8, n) if n > 1 else wl.csr_from_pairs(1, np.empty(0, np.int64), np.empty(0, np.int64))
    e = np.random.default_rng(m).integers(0, n, (m, 2)).astype(np.int32)
    src = np.repeat(np.arange(n), np.diff(ip))
    before = oracle.closure(n, ip, ix)
    want = oracle.closure(n, *wl.csr_from_pairs(n, np.concatenate([src, e[:, 0]]), np.concatenate([ix, e[:, 1]])))
    packed = fmt == pkg.BMLP_FMT_PACKED64
    mat = torch.from_numpy(wl.pack_rows(before).view(np.int64) if packed else before.astype(np.uint8)).cuda()
    with pkg.Context(0) as ctx:
        ctx.insert(mat, n, e, fmt=fmt)
        assert ctx.stats()["iterations"] == m
        torch.cuda.synchronize()
    got = mat.cpu().numpy()
    np.testing.assert_array_equal(wl.unpack_rows(got.view(np.uint64), n) if packed else got, want)


@pytest.mark.parametrize("n,chunk", [(8192, 4), (8193, 3)])
def test_single_facts_take_no_workspace(n, chunk):
    mat = torch.zeros((n, (n + 63) // 64), dtype=torch.int64, device="cuda")
    ctxs, free = [pkg.Context(0) for _ in range(12)], {}  # a chunk's scratch is 1.2 MB of each context
    for m in (2, 3, 4):
        for ctx in ctxs:
            ctx.insert(mat, n, np.array([[k, k + 1] for k in range(m)], np.int32), fmt=pkg.BMLP_FMT_PACKED64)
        torch.cuda.synchronize()
        free[m] = torch.cuda.mem_get_info()[0]
    for ctx in ctxs:
        ctx.close()
    assert free[2] > free[4] and free[3] == free[2 if chunk > 3 else 4]
