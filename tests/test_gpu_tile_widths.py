"""Batches of the tiled frontiers at the numbers of reached constants where a batch narrows: up to 28,288 of them the frontier
of 64 rows fits an SM's shared memory (and 64 rows are taken where 32 would need twice the rounds), up to 55,616 that of 32;
and relations of which few constants have facts, many each. Rows and levels against the oracle's search."""
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


def reached(n, n1, d, seed, every=1):
    """n constants, exactly n1 of which facts point at; one in `every` constants has facts, d on average"""
    rng = np.random.default_rng(seed)
    label = rng.permutation(n)
    src = rng.integers(0, n // every, int(n // every * d)) * every
    dst = rng.integers(0, n1, len(src))
    src = np.concatenate([src, rng.integers(0, n // every, n1) * every])
    dst = np.concatenate([dst, np.arange(n1)])
    return wl.csr_from_pairs(n, label[src], label[dst])


def rows_on_device(n, csr):
    i = torch.repeat_interleave(torch.arange(n), torch.from_numpy(np.diff(csr[0]).astype(np.int64))).cuda()
    j = torch.from_numpy(np.asarray(csr[1], np.int64)).cuda()
    R = torch.zeros(n * wl.words(n), dtype=torch.int64, device="cuda")
    R.index_add_(0, i * wl.words(n) + (j >> 6), torch.ones_like(j) << (j & 63))
    return R


@pytest.mark.parametrize("n,n1,d,q,every", [(28400, 28288, 3.0, 4900, 1), (28400, 28289, 3.0, 4900, 1), (28289, 28289, 3.0, 130, 1),
                                            (55700, 55616, 3.0, 200, 1), (55700, 55617, 3.0, 200, 1), (65536, 65536, 3.0, 90, 1),
                                            (40000, 39000, 60.0, 300, 10), (9001, 8000, 12.0, 131, 4)])
def test_widths(ctx, n, n1, d, q, every):
    csr = reached(n, n1, d, n1 + q, every)
    src = wl.query_rows(n, q, 1, 3, 3).copy()
    src[q // 2] = 0
    want, levels = oracle.smp(n, *csr, src)
    s = torch.from_numpy(src.view(np.int64)).cuda()
    out = torch.full_like(s, -1)
    R = rows_on_device(n, csr)
    assert ctx.smp(R, n, s, q, out, fmt=PACKED) == int(levels.max()) + 1
    torch.cuda.synchronize()
    assert ctx.stats()["sliced_closures"] == 1
    np.testing.assert_array_equal(out.cpu().numpy().view(np.uint64), wl.pack_rows(want))
