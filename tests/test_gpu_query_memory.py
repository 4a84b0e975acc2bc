"""Query rows that stop on the way, where the device has no room for the word indexes that they would go on over: those rows are
expanded to their ends without them, the finished ones are left as they are."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pkg = pytest.importorskip("paper_2408_10369_gb300")

pytestmark = pytest.mark.gpu


def relation(n):
    """Two paths of 2,000 and 700 constants, and pairs."""
    k = np.arange(n - 1)
    one = np.where(k < 2700, (k != 1999) & (k != 2699), k % 2 == 0)
    return wl.csr_from_pairs(n, k[one], k[one] + 1)


@pytest.mark.parametrize("n,fmt", [(50000, pkg.BMLP_FMT_PACKED64), (65536, pkg.BMLP_FMT_PACKED64), (30001, pkg.BMLP_FMT_U8)])
@pytest.mark.parametrize("reflexive,in_place", [(False, False), (True, False), (True, True)])
def test_rows_that_stop_without_room_for_indexes(n, fmt, reflexive, in_place):
    csr = relation(n)
    packed = fmt == pkg.BMLP_FMT_PACKED64
    host = wl.csr_to_packed(n, *csr)
    R = torch.from_numpy(host.view(np.int64) if packed else wl.unpack_rows(host, n).astype(np.uint8)).cuda()
    rows = np.zeros((6, n), bool)
    for r, at in enumerate(([0], [2000], [2704], [], [5, 2704, 2710], [1999, n - 1])):
        rows[r, at] = True
    src = wl.pack_rows(rows)
    want, levels = oracle.smp(n, *csr, src)
    want = wl.pack_rows(want) | (src if reflexive else 0)
    s = torch.from_numpy(src.view(np.int64)).cuda()
    out = s if in_place else torch.full_like(s, -1)
    spare = n * n // 8 + (64 << 20) if not packed else 64 << 20  # bytes become bit rows first
    with pkg.Context(0) as ctx:
        torch.cuda.synchronize()
        held = torch.empty(torch.cuda.mem_get_info()[0] - spare - (32 << 20), dtype=torch.uint8, device="cuda")
        try:
            it = ctx.smp(R, n, s, len(src), out, fmt=fmt, reflexive=reflexive, variant="smp_packed")
            torch.cuda.synchronize()
        finally:
            del held
            torch.cuda.empty_cache()
        assert it == int(levels.max()) + 1
        np.testing.assert_array_equal(out.cpu().numpy().view(np.uint64), want)
        assert ctx.stats()["product_launches"] == 2  # some rows stopped
