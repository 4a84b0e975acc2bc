"""A few query rows expanded straight from R's rows (one cluster per row): sizes around the words, shares and passes of the
kernel, both cluster sizes, long paths, dense rows, dirty padding bits, empty rows, reflexive and in-place results, against
the oracle's search; and the same rows through the batch kernels."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pkg = pytest.importorskip("paper_2408_10369_gb300")
from paper_2408_10369_gb300 import bmlp  # noqa: E402

pytestmark = pytest.mark.gpu
PACKED = bmlp.BMLP_FMT_PACKED64


@pytest.fixture(scope="module")
def ctx():
    c = pkg.Context(0)
    yield c
    c.close()


def relation(kind, n, d, seed):
    if kind == "chain":
        k = np.arange(n - 1)
        return wl.csr_from_pairs(n, k, k + 1)
    if kind == "cycle":
        k = np.arange(n)
        return wl.csr_from_pairs(n, k, (k + 1) % n)
    return wl.er_graph(n, d, seed)


def packed(n, ip, ix, dirty=False):
    P = wl.csr_to_packed(n, ip, ix).view(np.int64).copy()
    if dirty and n % 64:
        P[:, -1] |= np.int64(np.uint64(~((1 << (n % 64)) - 1) & 0xFFFFFFFFFFFFFFFF).view(np.int64))
    return torch.from_numpy(P).cuda()


@pytest.mark.parametrize("kind,n,d,q", [("er", 1, 0.0, 1), ("er", 2, 1.0, 2), ("er", 63, 1.5, 3), ("er", 64, 1.5, 5),
                                        ("er", 65, 30.0, 8), ("chain", 700, 0, 2), ("cycle", 130, 0, 4), ("er", 1000, 1.2, 9),
                                        ("er", 1025, 300.0, 10), ("er", 5000, 50.0, 1), ("er", 8193, 3.0, 17),
                                        ("er", 8200, 2.0, 18), ("er", 3000, 1.5, 37), ("er", 4100, 2.0, 63), ("er", 16385, 2.5, 2), ("er", 33000, 2.0, 3)])
@pytest.mark.parametrize("reflexive", [False, True])
def test_query_rows(ctx, kind, n, d, q, reflexive):
    ip, ix = relation(kind, n, d, n)
    src = wl.query_rows(n, q, 1, min(n, 3), 5).copy()
    if q > 2:
        src[1] = 0
    want, levels = oracle.smp(n, ip, ix, src)
    if reflexive:
        want = want | wl.unpack_rows(src, n)
    R = packed(n, ip, ix, dirty=True)
    s = torch.from_numpy(src.view(np.int64)).cuda()
    out = torch.full_like(s, -1)
    it = ctx.smp(R, n, s, q, out, fmt=PACKED, reflexive=reflexive)
    torch.cuda.synchronize()
    assert ctx.stats()["launches"] == 1  # no index was built
    np.testing.assert_array_equal(wl.unpack_rows(out.cpu().numpy().view(np.uint64), n), want)
    assert it == int(levels.max()) + 1
    assert n % 64 == 0 or not bool((out[:, -1].cpu().numpy().view(np.uint64) >> np.uint64(n % 64)).any())
    if not reflexive:
        ctx.smp(R, n, s, q, s, fmt=PACKED)  # in place
        assert torch.equal(s, out)


def test_query_rows_match_batches(ctx):
    """The same rows one by one and in a batch too large for one launch of clusters; byte matrices."""
    n, q = 4100, 70
    ip, ix = wl.er_graph(n, 3.0, 8)
    R = torch.from_numpy(wl.dense_u8(n, ip, ix)).cuda()
    src = torch.from_numpy(wl.query_rows(n, q, 1, 8, 9).view(np.int64)).cuda()
    batch, one = torch.zeros_like(src), torch.zeros_like(src)
    levels = ctx.smp(R, n, src, q, batch)
    assert ctx.stats()["launches"] > 2
    got = [ctx.smp(R, n, src[k:k + 1], 1, one[k:k + 1]) for k in range(q)]
    assert torch.equal(batch, one) and max(got) == levels


def test_query_rows_budget(ctx):
    n = 20000
    k = np.arange(n - 1)
    R = packed(n, *wl.csr_from_pairs(n, k, k + 1))
    src = torch.zeros((1, wl.words(n)), dtype=torch.int64, device="cuda")
    src[0, 0] = 1
    out = torch.zeros_like(src)
    with pytest.raises(pkg.BmlpError) as e:
        ctx.smp(R, n, src, 1, out, fmt=PACKED, budget_ns=50000)
    assert e.value.status == bmlp.BMLP_ERR_BUDGET
    assert ctx.smp(R, n, src, 1, out, fmt=PACKED) == n
