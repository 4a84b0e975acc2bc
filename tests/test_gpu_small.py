"""Closures and compositions of small relations in one launch: sizes at the edges of words, groups of lanes, rows a block
and of the whole range, dense, sparse and path-like relations, results over the operand, an exhausted limit of products
and an exhausted wait, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pkg = pytest.importorskip("paper_2408_10369_gb300")
from paper_2408_10369_gb300 import bmlp  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = pkg.Context(0)
    yield c
    c.close()


def relation(kind, n, seed):
    if kind == "path":
        p = np.random.default_rng(seed).permutation(n)
        return wl.csr_from_pairs(n, p[:-1], p[1:])
    return wl.er_graph(n, {"er": min(2.0, n / 2), "dense": n * 0.5, "empty": 0.0}[kind], seed)


def operand(n, csr, fmt):
    if fmt == "packed":
        return torch.from_numpy(wl.csr_to_packed(n, *csr).view(np.int64)).cuda()
    return torch.from_numpy(wl.dense_u8(n, *csr)).cuda()


def bits(t, n, fmt):
    return wl.unpack_rows(t.cpu().numpy().view(np.uint64), n) if fmt == "packed" else t.cpu().numpy()


FMT = {"u8": bmlp.BMLP_FMT_U8, "packed": bmlp.BMLP_FMT_PACKED64}


@pytest.mark.parametrize("n", [1, 2, 31, 33, 64, 127, 129, 256, 257, 303, 305, 512, 513, 609, 1000, 1023, 1024, 1025])
@pytest.mark.parametrize("fmt", ["u8", "packed"])
def test_closures(ctx, n, fmt):
    for kind in ("er", "dense", "empty") + (("path",) if n > 1 else ()):
        csr = relation(kind, n, n)
        want = oracle.closure(n, *csr)
        L = oracle.longest_shortest_path(n, *csr)
        for reflexive in (False, True):
            R = operand(n, csr, fmt)
            it = ctx.rms(R, n, R, fmt=FMT[fmt], reflexive=reflexive)  # in place
            ref = want.copy()
            if reflexive:
                np.fill_diagonal(ref, 1)
            np.testing.assert_array_equal(bits(R, n, fmt), ref)
            st = ctx.stats()
            assert it == oracle.rms_iterations(L) == st["product_launches"]
            assert st["e2m1_products"] == (0 if n <= 1024 else it)


@pytest.mark.parametrize("n", [1, 40, 257, 640, 1024])
@pytest.mark.parametrize("fmt", ["u8", "packed"])
def test_compositions(ctx, n, fmt):
    for k1, k2 in (("er", "er"), ("dense", "er"), ("er", "empty")):
        a, b = relation(k1, n, 3), relation(k2, n, 4)
        A, B = operand(n, a, fmt), operand(n, b, fmt)
        want = oracle.compose_rows(n, a, b)
        for out in (torch.empty_like(A), A):
            it = ctx.compose(A, B, n, out, fmt=FMT[fmt])
            np.testing.assert_array_equal(bits(out, n, fmt), want)
            assert it == oracle.rms_iterations(oracle.longest_shortest_path(n, *b))


def test_limits(ctx):
    n = 400
    csr = relation("path", n, 9)
    R, out = operand(n, csr, "u8"), torch.zeros((n, n), dtype=torch.uint8, device="cuda")
    for kwargs, status in (({"max_iters": 3}, bmlp.BMLP_ERR_NOT_CONVERGED), ({"timeout_ns": 1}, bmlp.BMLP_ERR_TIMEOUT)):
        with pytest.raises(bmlp.BmlpError) as e:
            ctx.rms(R, n, out, **kwargs)
        assert e.value.status == status
        assert ctx.rms(R, n, out) == oracle.rms_iterations(n - 1)
        np.testing.assert_array_equal(out.cpu().numpy(), oracle.closure(n, *csr))
