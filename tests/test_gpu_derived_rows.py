"""Frontier closures in which most rows follow from another row: chains of constants with one fact each (shorter and longer
than a row is derived over, into a core, into a constant without facts, into a cycle), rings whose deepest constants lie
on such a chain, self loops, and sources that nothing reaches, against the oracle's search: rows and level counts."""
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


def relation(n, core, gadgets, seed):
    """A random core on the first `core` constants (5 facts each), gadgets behind it, the numbers shuffled. The constants
    left over have one fact into the core (and nothing reaches them)."""
    ip, ix = wl.er_graph(core, 5.0, seed)
    pairs = [(i, int(j)) for i in range(core) for j in ix[ip[i]:ip[i + 1]]]
    at = core
    for kind, length in gadgets:
        chain = list(range(at, at + length))
        at += length
        pairs += list(zip(chain[:-1], chain[1:]))
        if kind == "core":
            pairs.append((chain[-1], 7))
        elif kind == "cycle":
            pairs.append((chain[-1], chain[0]))
        elif kind == "self":
            pairs.append((chain[-1], chain[-1]))
        elif kind == "ring":  # the first constant has a second fact, to a constant without facts
            pairs += [(chain[-1], chain[0]), (chain[0], at)]
            at += 1
        elif kind == "leaf":
            at += 1
            pairs.append((chain[-1], at - 1))
    pairs += [(i, i % core) for i in range(at, n)]
    p = np.random.default_rng(seed).permutation(n)
    src, dst = np.asarray(pairs, np.int64).T
    return wl.csr_from_pairs(n, p[src], p[dst])


@pytest.mark.parametrize("n,core,gadgets", [
    (4100, 3000, [("core", 5), ("core", 32), ("leaf", 3), ("self", 2), ("cycle", 4)]),
    (4200, 3000, [("core", 40), ("leaf", 33), ("leaf", 50), ("cycle", 60), ("ring", 6)]),
    (4200, 3000, [("ring", 30), ("ring", 12), ("cycle", 20)]),      # a ring's rows only look the deepest
    (5003, 2500, [("ring", 33), ("core", 31), ("ring", 45)]),
    (9000, 8990, []), (4097, 60, [("ring", 25)])])
def test_closures(ctx, n, core, gadgets):
    ip, ix = relation(n, core, gadgets, n + len(gadgets))
    P = torch.from_numpy(wl.csr_to_packed(n, ip, ix).view(np.int64)).cuda()
    rows = np.arange(n, dtype=np.int32)
    want, depth, _ = oracle.reach_rows(n, ip, ix, rows)
    for kwargs in ({}, {"budget_ns": 10**10}):  # under a budget every row is expanded
        out = torch.full_like(P, -1)
        it = ctx.rms(P, n, out, fmt=PACKED, variant="smp_packed", **kwargs)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(wl.unpack_rows(out.cpu().numpy().view(np.uint64), n), want)
        if ctx.stats()["frontier_squarings"] == 0:
            assert it == int(depth.max()) + 1
    if core > 2000:
        assert ctx.stats()["sliced_closures"] == 1


@pytest.mark.parametrize("n,q", [(4100, 70), (30000, 400), (65536, 150)])
def test_unreached_sources(ctx, n, q):
    ip, ix = relation(n, n // 2, [("core", 9)], n)
    src = wl.query_rows(n, q, 1, 12, 5).copy()
    src[1] = ~np.uint64(0)
    src[1, -1] >>= np.uint64(-n % 64)
    src[q // 2] = 0
    want, levels = oracle.smp(n, ip, ix, src)
    P = torch.from_numpy(wl.csr_to_packed(n, ip, ix).view(np.int64)).cuda()
    s = torch.from_numpy(src.view(np.int64)).cuda()
    for reflexive in (False, True):
        out = torch.full_like(s, -1)
        it = ctx.smp(P, n, s, q, out, fmt=PACKED, reflexive=reflexive)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(out.cpu().numpy().view(np.uint64), wl.pack_rows(want) | (src if reflexive else 0))
        assert it == int(levels.max()) + 1
