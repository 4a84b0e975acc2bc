"""Sliced frontiers with the frontier in shared memory: heavy in-lists (hubs, dense relations), constants that nothing
reaches, the sizes where the words narrow to 32 and 16 rows, batches that end inside a word, and budgets, against the
oracle's search."""
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
    rng = np.random.default_rng(seed)
    ip, ix = wl.er_graph(n, d, seed)
    src, dst = np.repeat(np.arange(n), np.diff(ip)), np.asarray(ix, np.int64)
    if kind == "hubs":  # a third of the facts end in 40 constants, and 100 constants have no fact pointing at them
        hub = rng.random(len(dst)) < 0.33
        dst = np.where(hub, 100 + rng.integers(0, 40, len(dst)), dst)
        dst = np.where(dst < 100, dst + 200, dst)
    if kind == "mixed":  # only one constant in twenty has facts, many of them
        keep = src % 20 == 0
        src, dst = src[keep], dst[keep]
    return wl.csr_from_pairs(n, src, dst)


@pytest.mark.parametrize("kind,n,d,q", [("er", 4096, 5.0, 64), ("er", 4099, 6.0, 65), ("mixed", 9001, 70.0, 131),
                                        ("mixed", 20000, 200.0, 1000), ("hubs", 5003, 6.0, 100), ("hubs", 9000, 8.0, 2500),
                                        ("er", 28671, 4.0, 600), ("er", 28737, 4.0, 600), ("hubs", 57345, 5.0, 200),
                                        ("er", 65535, 4.0, 300)])
def test_tile_batches(ctx, kind, n, d, q):
    ip, ix = relation(kind, n, d, n)
    src = wl.query_rows(n, q, 1, 8, 3).copy()
    src[q // 3] = 0
    want, levels = oracle.smp(n, ip, ix, src)
    P = torch.from_numpy(wl.csr_to_packed(n, ip, ix).view(np.int64)).cuda()
    s = torch.from_numpy(src.view(np.int64)).cuda()
    for reflexive in (False, True):
        out = torch.full_like(s, -1)
        it = ctx.smp(P, n, s, q, out, fmt=PACKED, reflexive=reflexive)
        torch.cuda.synchronize()
        assert kind == "mixed" or ctx.stats()["sliced_closures"] == 1
        np.testing.assert_array_equal(out.cpu().numpy().view(np.uint64), wl.pack_rows(want) | (src if reflexive else 0))
        assert it == int(levels.max()) + 1


@pytest.mark.parametrize("kind,n,d", [("hubs", 4500, 6.0), ("mixed", 4100, 100.0), ("hubs", 30011, 5.0)])
def test_tile_closures(ctx, kind, n, d):
    ip, ix = relation(kind, n, d, 7)
    P = torch.from_numpy(wl.csr_to_packed(n, ip, ix).view(np.int64)).cuda()
    out = torch.zeros_like(P)
    it = ctx.rms(P, n, out, fmt=PACKED, variant="smp_packed")
    torch.cuda.synchronize()
    sliced = ctx.stats()["sliced_closures"]  # (rows of "mixed" widen too slowly: squared first, so other levels)
    assert sliced == (kind != "mixed")
    rows = np.arange(n, dtype=np.int32) if n < 10000 else np.unique(np.linspace(0, n - 1, 400).astype(np.int32))
    want, depth, _ = oracle.reach_rows(n, ip, ix, rows)
    np.testing.assert_array_equal(wl.unpack_rows(out.cpu().numpy().view(np.uint64)[rows], n), want)
    if sliced:
        assert it >= int(depth.max()) + 1 and (n >= 10000 or it == int(depth.max()) + 1)
