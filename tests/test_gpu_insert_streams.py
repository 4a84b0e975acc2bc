"""Insertions whose launches are still running when the next one comes: on other streams of one context (the calls share the
context's workspace), and recorded in a graph that is replayed after the facts' host memory is gone."""
import gc

import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pkg = pytest.importorskip("paper_2408_10369_gb300")

pytestmark = pytest.mark.gpu
PACKED = pkg.BMLP_FMT_PACKED64


def grown(n, d, m, seed):
    """(closure as packed rows, m new facts, the closure of both as bytes)"""
    ip, ix = wl.er_graph(n, d, seed)
    e = np.random.default_rng(seed).integers(0, n, (m, 2)).astype(np.int32)
    src = np.repeat(np.arange(n), np.diff(ip))
    want = oracle.closure(n, *wl.csr_from_pairs(n, np.concatenate([src, e[:, 0]]), np.concatenate([ix, e[:, 1]])))
    return torch.from_numpy(wl.pack_rows(oracle.closure(n, ip, ix)).view(np.int64)).cuda(), e, want


def test_insertions_on_streams_of_one_context():
    cases = [grown(4000, 0.6, 1500, 1), grown(700, 0.8, 40, 2), grown(2500, 0.5, 1024, 3)]
    ctx = pkg.Context(0)
    try:
        streams = [torch.cuda.Stream() for _ in cases]
        for first in range(6):  # the workspaces grow in the first round
            mats = [c.clone() for c, _, _ in cases]
            torch.cuda.synchronize()
            for k in range(len(cases)):
                k = (k + first) % len(cases)
                ctx.insert(mats[k], len(mats[k]), cases[k][1], fmt=PACKED, stream=streams[k])
            torch.cuda.synchronize()
            for got, (_, _, want) in zip(mats, cases):
                np.testing.assert_array_equal(wl.unpack_rows(got.cpu().numpy().view(np.uint64), len(got)), want)
    finally:
        ctx.close()


@pytest.mark.parametrize("m", [2, 3, 300])
def test_insertion_in_a_graph(m):
    n = 1100
    before, e, want = grown(n, 0.7, m, 4)
    other, e2, want2 = grown(900, 0.7, 500, 5)
    ctx = pkg.Context(0)
    try:
        mat, stream = before.clone(), torch.cuda.Stream()
        facts = e.copy()
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            ctx.insert(mat, n, facts, fmt=PACKED, stream=stream)
        assert torch.equal(mat, before)
        facts[:] = 0
        del facts
        gc.collect()
        ctx.insert(other, 900, e2, fmt=PACKED)  # takes the workspaces
        graph.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(wl.unpack_rows(mat.cpu().numpy().view(np.uint64), n), want)
        np.testing.assert_array_equal(wl.unpack_rows(other.cpu().numpy().view(np.uint64), 900), want2)
    finally:
        ctx.close()
