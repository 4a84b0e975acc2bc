"""A squaring whose restricted form stops with zeros open, and which a product over a slice of the constants then fills: the
slice is judged by its own completion, so no whole product follows."""
import torch
import pytest

pkg = pytest.importorskip("paper_2408_10369_gb300")
from paper_2408_10369_gb300 import bmlp  # noqa: E402

pytestmark = pytest.mark.gpu


def test_slice_after_an_open_restricted_squaring():
    # Every constant has facts with all others, with these exceptions: only the last 100 (T) have a fact
    # with z = 1500, and the first 801 (A) have no facts with T. After one squaring all entries are set but (A, z): rows
    # of A name 801 rows of A before the first one that has z, more than a restricted squaring reads of a dense row, and a
    # slice of the first 1,024 constants includes 223 that have it.
    n, z = 9216, 1500
    R = torch.ones((n, n), dtype=torch.uint8, device="cuda")
    R[:, z] = 0
    R[n - 100:, z] = 1
    R[:801, n - 100:] = 0
    out = torch.zeros_like(R)
    with pkg.Context(0) as ctx:
        it = ctx.rms(R, n, out, variant="rms_tc")
        torch.cuda.synchronize()
        st = ctx.stats()
    assert bool((out == 1).all())
    assert it == 3
    assert st["e2m1_products"] == 1 and st["thin_squarings"] == 2
