"""Squarings that start with a product over a slice of the constants: completed on the rows and columns that still hold
zeros where those are few, and by the rest of the product where they are many (an acyclic relation: half of the closure
stays zero). Bits and product counts against the oracle."""
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


def relation(kind, n, d, seed):
    ip, ix = wl.er_graph(n, d, seed)
    if kind == "er":
        return ip, ix
    src, dst = np.repeat(np.arange(n), np.diff(ip)), np.asarray(ix)
    if kind == "dag":
        return wl.csr_from_pairs(n, np.minimum(src, dst), np.maximum(src, dst))
    # a quarter of the constants form a dense core, the others reach it or are reached from it only
    core = n // 4
    a, b = src % core, dst % core
    out = src[: n] % n
    return wl.csr_from_pairs(n, np.concatenate([a, np.arange(core, n // 2), np.zeros(n - n // 2, np.int64) + out[n // 2:] % core]),
                             np.concatenate([b, np.arange(core, n // 2) % core, np.arange(n // 2, n)]))


@pytest.mark.parametrize("kind,n,d,seed", [("er", 8193, 3.0, 1), ("er", 12000, 4.0, 2), ("er", 16111, 2.2, 3),
                                           ("dag", 8200, 4.0, 4), ("dag", 12289, 6.0, 5), ("core", 9999, 5.0, 6)])
@pytest.mark.parametrize("fmt,reflexive", [("packed", False), ("u8", True)])
def test_sliced_squarings(ctx, kind, n, d, seed, fmt, reflexive):
    ip, ix = relation(kind, n, d, seed)
    want = oracle.closure(n, ip, ix)
    iters = oracle.rms_iterations(oracle.longest_shortest_path(n, ip, ix))
    if reflexive:
        np.fill_diagonal(want, 1)
    if fmt == "packed":
        R = torch.from_numpy(wl.csr_to_packed(n, ip, ix).view(np.int64)).cuda()
        out = torch.zeros_like(R)
        it = ctx.rms(R, n, out, fmt=bmlp.BMLP_FMT_PACKED64, variant="rms_tc", reflexive=reflexive)
        got = wl.unpack_rows(out.cpu().numpy().view(np.uint64), n)
    else:
        R = torch.from_numpy(wl.dense_u8(n, ip, ix)).cuda()
        out = torch.zeros_like(R)
        it = ctx.rms(R, n, out, variant="rms_tc", reflexive=reflexive)
        got = out.cpu().numpy()
    np.testing.assert_array_equal(got, want)
    st = ctx.stats()
    assert it == iters == st["sparse_squarings"] + st["product_launches"] + st["thin_squarings"]
