"""Packed compositions of few constants: the whole-row product is cheaper there than the predicted fixed cost of the one over
word indexes, so that none is built for the choice and the host does not wait for its cost."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pkg = pytest.importorskip("paper_2408_10369_gb300")
from paper_2408_10369_gb300 import bmlp  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d1,d2", [(400, 3.0, 0.0), (400, 2.0, 0.5), (3000, 3.0, 0.0), (4300, 2.0, 0.6)])
def test_small_packed_compositions(n, d1, d2):
    a, b = wl.er_graph(n, d1, 1), wl.er_graph(n, d2, 2)
    A, B = (torch.from_numpy(wl.csr_to_packed(n, *x).view(np.int64)).cuda() for x in (a, b))
    out = torch.zeros_like(A)
    with pkg.Context(0) as ctx:
        it = ctx.compose(A, B, n, out, fmt=bmlp.BMLP_FMT_PACKED64, variant="rms_packed")
        torch.cuda.synchronize()
        assert ctx.stats()["host_syncs"] == it + 2  # the first index's words, every squaring, the product
    np.testing.assert_array_equal(wl.unpack_rows(out.cpu().numpy().view(np.uint64), n), oracle.compose_rows(n, a, b))
