"""Compositions (I + R2+) R1 formed from bit rows: R1 sparse (row ORs of the transposed closure) and dense (a product on
the tensor cores), R2's closure sparse, dense by a sliced squaring, or reached without a squaring, in bytes and bit rows,
at sizes around the line of 4,096 constants, with n odd and a multiple of 64, against the oracle."""
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


def operand(n, csr, fmt):
    if fmt == "packed":
        return torch.from_numpy(wl.csr_to_packed(n, *csr).view(np.int64)).cuda()
    return torch.from_numpy(wl.dense_u8(n, *csr)).cuda()


# products: on the tensor cores (1 more than the closure's) or by row ORs
@pytest.mark.parametrize("n,d1,d2,rows", [(4095, 2.0, 3.0, None), (4097, 2.0, 3.0, True), (4097, 400.0, 3.0, False),
                                          (4160, 0.0, 3.0, True), (6001, 3.0, 0.5, True), (6016, 2.0, 0.0, True),
                                          (8193, 2.0, 4.0, True), (9001, 700.0, 2.0, False)])
@pytest.mark.parametrize("fmt", ["u8", "packed"])
def test_compose(ctx, n, d1, d2, rows, fmt):
    a, b = wl.er_graph(n, d1, n), wl.er_graph(n, d2, n + 1)
    f = bmlp.BMLP_FMT_PACKED64 if fmt == "packed" else bmlp.BMLP_FMT_U8
    A, B = operand(n, a, fmt), operand(n, b, fmt)
    out = torch.full_like(A, 1)
    it = ctx.compose(A, B, n, out, fmt=f, variant="rms_tc")
    st = ctx.stats()
    got = out.cpu().numpy()
    got = wl.unpack_rows(got.view(np.uint64), n) if fmt == "packed" else got
    np.testing.assert_array_equal(got, oracle.compose_rows(n, a, b))
    assert it == oracle.rms_iterations(oracle.longest_shortest_path(n, *b))
    if rows is not None:  # the composition's own product is one of product_launches either way
        on_tc = st["e2m1_products"] - (st["product_launches"] - 1) == 1
        assert on_tc == (not rows)
