"""Frontier closures of relations in which most rows are one fact, a step or more from a few rows with several: the level count
of a row one step away is certain, also where the deepest constants of the other row lie one step before it or are its own."""
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


def relation(kind, n, seed):
    g = np.random.default_rng(seed)
    k = np.arange(1, n)
    if kind == "star":    # the hub's own row ends at the hub alone
        src, dst = np.concatenate([k, 0 * k]), np.concatenate([0 * k, k])
    elif kind == "self":  # all to a constant with itself and one other
        src, dst = np.concatenate([k, [0, 0]]), np.concatenate([0 * k, [0, 1]])
    elif kind == "loop":  # all to a constant, which comes back to itself after three steps; a leaf is its second fact
        src, dst = np.concatenate([k[3:], [0, 1, 2, 0]]), np.concatenate([0 * k[3:], [1, 2, 0, 3]])
    else:                 # `kind` hubs of many facts; the others one each: to a hub, to another (chains, cycles), to themselves
        to = np.where(g.random(n) < 0.6, g.integers(0, kind, n), g.integers(0, n, n))
        src = np.concatenate([np.arange(kind, n), np.repeat(np.arange(kind), n // 3)])
        dst = np.concatenate([to[kind:], g.integers(0, n, kind * (n // 3))])
    p = g.permutation(n)
    return wl.csr_from_pairs(n, p[src], p[dst])


@pytest.mark.parametrize("kind,n", [("star", 4097), ("self", 4200), ("loop", 4200), ("loop", 9001)] +
                         [(h, n) for h in (1, 2, 3, 40) for n in (4099, 4600, 6001)])
def test_level_counts(kind, n):
    ip, ix = relation(kind, n, n)
    R = torch.from_numpy(wl.csr_to_packed(n, ip, ix).view(np.int64)).cuda()
    want, depth, _ = oracle.reach_rows(n, ip, ix, np.arange(n, dtype=np.int32))
    with pkg.Context(0) as ctx:
        for kwargs in ({}, {"budget_ns": 10**10}):  # under a budget every row is expanded
            out = torch.full_like(R, -1)
            it = ctx.rms(R, n, out, fmt=PACKED, variant="smp_packed", **kwargs)
            torch.cuda.synchronize()
            np.testing.assert_array_equal(wl.unpack_rows(out.cpu().numpy().view(np.uint64), n), want)
            if ctx.stats()["frontier_squarings"] == 0:
                assert it == int(depth.max()) + 1


def test_rows_one_step_from_a_hub_are_not_expanded():
    n = 30000
    R = torch.from_numpy(wl.csr_to_packed(n, *relation("star", n, 1)).view(np.int64)).cuda()
    out, best = torch.zeros_like(R), 1e9
    with pkg.Context(0) as ctx:
        for _ in range(8):
            torch.cuda.synchronize()
            t = time.perf_counter()
            assert ctx.rms(R, n, out, fmt=PACKED, variant="smp_packed") == 3
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
    assert bool((out == out[0]).all())
    assert best < 1.2e-3  # 0.8 ms; 1.6 ms with those rows expanded
