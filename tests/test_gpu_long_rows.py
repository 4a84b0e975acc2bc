"""Relations in which a few rows or columns have hundreds of times the mean of facts: such rows are walked by a whole block
of the passes over a word index (products, their costs, the lists of a frontier). Rows at the edge of 64 nonzero words,
more of them than a block's queue holds, and rows that name each other, against the oracle."""
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


def relation(n, rows, words, seed):
    """One fact a row on average, and `rows` rows of one fact in each of `words` nonzero words (as many as n has at most)."""
    rng = np.random.default_rng(seed)
    ip, ix = wl.er_graph(n, 1.0, seed)
    src, dst = np.repeat(np.arange(n), np.diff(ip)), np.asarray(ix, np.int64)
    at = rng.choice(n, rows, replace=False)
    w = min(words, n // 64)
    col = np.concatenate([64 * rng.choice(n // 64, w, replace=False) + rng.integers(0, 64, w) for _ in range(rows)])
    return wl.csr_from_pairs(n, np.concatenate([src, np.repeat(at, w)]), np.concatenate([dst, col]))


@pytest.mark.parametrize("n,rows,words", [(4225, 3, 64), (4225, 3, 65), (4225, 400, 66), (9001, 12, 140), (14541, 1, 227)])
def test_products(ctx, n, rows, words):
    a, b = relation(n, rows, words, 1), relation(n, rows, words, 2)
    A, B = (torch.from_numpy(wl.csr_to_packed(n, *x).view(np.int64)).cuda() for x in (a, b))
    out = torch.zeros_like(A)
    ctx.compose(A, B, n, out, fmt=PACKED)
    got = wl.unpack_rows(out.cpu().numpy().view(np.uint64), n)
    np.testing.assert_array_equal(got, oracle.compose_rows(n, a, b))


@pytest.mark.parametrize("variant", ["rms_tc", "smp_packed"])
@pytest.mark.parametrize("n,rows,words", [(4225, 2, 65), (4225, 2500, 66), (9001, 12, 140)])
@pytest.mark.parametrize("transposed", [False, True])
def test_closures(ctx, variant, n, rows, words, transposed):
    ip, ix = relation(n, rows, words, 3)
    if transposed:
        ip, ix = wl.csr_from_pairs(n, np.asarray(ix, np.int64), np.repeat(np.arange(n), np.diff(ip)))
    P = torch.from_numpy(wl.csr_to_packed(n, ip, ix).view(np.int64)).cuda()
    out = torch.zeros_like(P)
    it = ctx.rms(P, n, out, fmt=PACKED, variant=variant)
    np.testing.assert_array_equal(wl.unpack_rows(out.cpu().numpy().view(np.uint64), n), oracle.closure(n, ip, ix))
    if variant == "rms_tc":
        assert it == oracle.rms_iterations(oracle.longest_shortest_path(n, ip, ix))
