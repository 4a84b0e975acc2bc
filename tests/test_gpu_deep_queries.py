"""Query rows whose frontier is narrow for many levels, or that cost more from R's rows than over word indexes: exact rows and
levels whichever form ends them, against the oracle's search or what the relation says, and the time of a path."""
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


@pytest.fixture(scope="module")
def ctx():
    c = pkg.Context(0)
    yield c
    c.close()


def relation(kind, n, seed):
    k = np.arange(n)
    p = np.random.default_rng(seed).permutation(n)
    if kind == "path":
        return wl.csr_from_pairs(n, p[:-1], p[1:])
    if kind == "cycle":
        return wl.csr_from_pairs(n, p, np.roll(p, -1))
    if kind == "beads":  # a path of 2/3 of the constants, every 40th of them also with facts to a bunch of 30 others that meet again
        m = 2 * n // 3
        i, j = [k[:m - 1]], [k[1:m]]
        bunch = m + np.arange((n - m) // 30 * 30).reshape(-1, 30)
        at = 40 * np.arange(len(bunch)) % (m - 45)
        i += [np.repeat(at, 30), bunch.ravel()]
        j += [bunch.ravel(), np.repeat(at + 43, 30)]
        return wl.csr_from_pairs(n, p[np.concatenate(i)], p[np.concatenate(j)])
    if kind == "grid":
        side = int(n ** 0.5)
        right, down = k[(k % side != side - 1) & (k + 1 < n)], k[k + side < n]
        return wl.csr_from_pairs(n, np.concatenate([right, down]), np.concatenate([right + 1, down + side]))
    return wl.er_graph(n, float(kind[2:]), seed)


@pytest.mark.parametrize("kind,n,q", [("path", 40, 2), ("path", 64, 1), ("path", 65, 5), ("cycle", 700, 3), ("path", 2047, 1),
                                      ("beads", 1500, 4), ("beads", 6000, 17), ("cycle", 8191, 2), ("path", 8192, 9),
                                      ("path", 8193, 1), ("beads", 8200, 30), ("cycle", 9001, 63), ("grid", 4000, 7),
                                      ("grid", 9000, 19), ("grid", 20011, 40), ("er1.1", 20000, 63), ("er1.02", 7000, 20)])
@pytest.mark.parametrize("reflexive", [False, True])
@pytest.mark.parametrize("fmt", ["packed", "u8"])
def test_deep_rows(ctx, kind, n, q, reflexive, fmt):
    ip, ix = relation(kind, n, n)
    src = wl.query_rows(n, q, 1, 2, 5).copy()
    if q > 2:
        src[1] = 0
    want, levels = oracle.smp(n, ip, ix, src)
    if reflexive:
        want = want | wl.unpack_rows(src, n)
    if fmt == "packed":
        P = wl.csr_to_packed(n, ip, ix).copy()
        if n % 64:  # bits beyond column n are ignored
            P[:, -1] |= np.uint64(~((1 << (n % 64)) - 1) & 0xFFFFFFFFFFFFFFFF)
        R = torch.from_numpy(P.view(np.int64)).cuda()
    else:
        R = torch.from_numpy(wl.dense_u8(n, ip, ix)).cuda()
    f = PACKED if fmt == "packed" else bmlp.BMLP_FMT_U8
    s = torch.from_numpy(src.view(np.int64)).cuda()
    out = torch.full_like(s, -1)
    for _ in range(2):
        assert ctx.smp(R, n, s, q, out, fmt=f, reflexive=reflexive) == int(levels.max()) + 1
        np.testing.assert_array_equal(out.cpu().numpy().view(np.uint64), wl.pack_rows(want))
    assert ctx.smp(R, n, s, q, s, fmt=f, reflexive=reflexive) == int(levels.max()) + 1  # in place
    assert torch.equal(s, out)
    if fmt == "packed":
        launches = ctx.stats()["launches"]
        assert launches == 1 if n <= 8192 else kind not in ("path", "cycle") or launches > 1


def test_wide_rows_on_a_large_relation(ctx):
    """63 rows that reach most of 80,000 constants (50 GB of rows of R): finished over the word indexes."""
    n, q = 80000, 63
    csr = wl.er_graph(n, 3.0, 2)
    i = torch.repeat_interleave(torch.arange(n), torch.from_numpy(np.diff(csr[0]).astype(np.int64))).cuda()
    j = torch.from_numpy(np.asarray(csr[1], np.int64)).cuda()
    R = torch.zeros(n * wl.words(n), dtype=torch.int64, device="cuda")
    R.index_add_(0, i * wl.words(n) + (j >> 6), torch.ones_like(j) << (j & 63))
    src = wl.query_rows(n, q, 1, 2, 5)
    want, levels = oracle.smp(n, *csr, src)
    s = torch.from_numpy(src.view(np.int64)).cuda()
    out = torch.full_like(s, -1)
    assert ctx.smp(R, n, s, q, out, fmt=PACKED) == int(levels.max()) + 1
    np.testing.assert_array_equal(out.cpu().numpy().view(np.uint64), wl.pack_rows(want))
    assert ctx.stats()["launches"] > 1


def test_limits_of_deep_rows(ctx):
    for n in (3000, 12000):
        k = np.arange(n - 1)
        R = torch.from_numpy(wl.csr_to_packed(n, *wl.csr_from_pairs(n, k, k + 1)).view(np.int64)).cuda()
        src = torch.zeros((2, wl.words(n)), dtype=torch.int64, device="cuda")
        src[:, 0] = 1
        out = torch.zeros_like(src)
        for opt, status in ((dict(max_iters=n - 1), bmlp.BMLP_ERR_NOT_CONVERGED), (dict(budget_ns=100000), bmlp.BMLP_ERR_BUDGET)):
            with pytest.raises(bmlp.BmlpError) as e:
                ctx.smp(R, n, src, 2, out, fmt=PACKED, **opt)
            assert e.value.status == status
        assert ctx.smp(R, n, src, 2, out, fmt=PACKED, max_iters=n) == n


@pytest.mark.parametrize("n", [500, 5000, 20000])
def test_time_of_a_path(ctx, n):
    """A level of a path takes 1.6 us over the word indexes, 0.6 us by one warp, and took 2.7 to 3.4 us by a cluster."""
    k = np.arange(n - 1)
    R = torch.from_numpy(wl.csr_to_packed(n, *wl.csr_from_pairs(n, k, k + 1)).view(np.int64)).cuda()
    src = torch.zeros((1, wl.words(n)), dtype=torch.int64, device="cuda")
    src[0, 0] = 1
    out = torch.zeros_like(src)
    best = 1e9
    for _ in range(6):
        torch.cuda.synchronize()
        t = time.perf_counter()
        assert ctx.smp(R, n, src, 1, out, fmt=PACKED) == n
        best = min(best, time.perf_counter() - t)
    assert best < 150e-6 + 2.0e-6 * n
