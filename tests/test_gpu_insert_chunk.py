"""Facts inserted in chunks: at the chunk's edges, as long chains and cycles of new facts that link to one another, and
over more facts than constants, against the oracle's closure of the grown relation."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pkg = pytest.importorskip("paper_2408_10369_gb300")

pytestmark = pytest.mark.gpu
PACKED = pkg.BMLP_FMT_PACKED64


@pytest.fixture(scope="module")
def ctx():
    c = pkg.Context(0)
    yield c
    c.close()


def facts(kind, n, m, rng):
    if kind == "random":
        return rng.integers(0, n, (m, 2))
    k = np.arange(m)
    e = np.stack([k % n, (k + 1) % n], 1)                   # a path (a cycle once m >= n)
    if kind == "star":
        e = np.where((k % 2 == 0)[:, None], np.stack([k % n, 0 * k], 1), np.stack([0 * k, k % n], 1))
    return e[rng.permutation(m)] if kind != "reverse" else e[::-1]


@pytest.mark.parametrize("kind", ["random", "path", "reverse", "star"])
@pytest.mark.parametrize("n,d,m", [(5, 0.0, 3), (97, 0.3, 31), (97, 0.3, 200), (640, 0.0, 64), (641, 0.5, 65),
                                   (1100, 0.2, 1024), (1500, 0.0, 1023), (1500, 0.4, 1025), (1300, 0.0, 2600)])
def test_chunks_match_recompute(ctx, kind, n, d, m):
    rng = np.random.default_rng(n + m)
    ip, ix = wl.er_graph(n, d, 5)
    e = np.ascontiguousarray(facts(kind, n, m, rng), np.int32)
    C = torch.zeros((n, wl.words(n)), dtype=torch.int64, device="cuda")
    ctx.rms(torch.from_numpy(wl.csr_to_packed(n, ip, ix).view(np.int64)).cuda(), n, C, fmt=PACKED)
    ctx.insert(C, n, torch.from_numpy(e).cuda(), fmt=PACKED)
    src = np.repeat(np.arange(n), np.diff(ip))
    want = oracle.closure(n, *wl.csr_from_pairs(n, np.concatenate([src, e[:, 0]]), np.concatenate([ix, e[:, 1]])))
    np.testing.assert_array_equal(wl.unpack_rows(C.cpu().numpy().view(np.uint64), n), want)
