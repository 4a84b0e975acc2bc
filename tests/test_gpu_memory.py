"""Calls on a device whose memory is mostly held by the caller: the forms that want more workspace give way to those that
need less, and a call that did not fit runs once there is room."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pkg = pytest.importorskip("paper_2408_10369_gb300")
from paper_2408_10369_gb300 import bmlp  # noqa: E402

pytestmark = pytest.mark.gpu
PACKED = bmlp.BMLP_FMT_PACKED64


def hold_all_but(free):
    """Device memory held so that about `free` bytes are left."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - free, dtype=torch.uint8, device="cuda")


@pytest.fixture(scope="module")
def large_problems():
    n = 12000
    csr = wl.er_graph(n, 3.0, 11)
    R = torch.from_numpy(wl.csr_to_packed(n, *csr).view(np.int64)).cuda()
    with pkg.Context(0) as ctx:  # kernels and graphs are loaded while there is room
        r = torch.from_numpy(wl.csr_to_packed(4096, *wl.er_graph(4096, 3.0, 1)).view(np.int64)).cuda()
        ctx.batch_run([dict(n=4096, R1=r, out=torch.zeros_like(r), fmt=PACKED) for _ in range(4)])
    return n, R, wl.pack_rows(oracle.closure(n, *csr))


def test_batch_branches_give_way_to_memory(large_problems):
    """Four problems of 12,000 constants on four branches take 1.9 GB of scratch, on two 1.0 GB."""
    n, R, want = large_problems
    outs = [torch.zeros_like(R) for _ in range(4)]
    with pkg.Context(0) as ctx:
        held = hold_all_but(1300 << 20)
        try:
            ctx.batch_run([dict(n=n, R1=R, out=o, fmt=PACKED) for o in outs])
            torch.cuda.synchronize()
        finally:
            del held
            torch.cuda.empty_cache()
    for o in outs:
        np.testing.assert_array_equal(o.cpu().numpy().view(np.uint64), want)


def test_batch_runs_once_there_is_room(large_problems):
    n, R, want = large_problems
    out = torch.zeros_like(R)
    items = pkg.Context.problems([dict(n=n, R1=R, out=out, fmt=PACKED)])
    with pkg.Context(0) as ctx:
        held = hold_all_but(200 << 20)
        try:
            for _ in range(2):
                with pytest.raises(bmlp.BmlpError) as e:
                    ctx.batch_run(items)
                assert e.value.status == bmlp.BMLP_ERR_OOM
        finally:
            del held
            torch.cuda.empty_cache()
        ctx.batch_run(items)
        torch.cuda.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy().view(np.uint64), want)


def workspace_of(R, n, out, **opt):
    """Bytes that a context takes for this closure, and its statistics."""
    out.zero_()
    torch.cuda.synchronize()
    with pkg.Context(0) as ctx:
        before = torch.cuda.mem_get_info()[0]
        ctx.rms(R, n, out, **opt)
        torch.cuda.synchronize()
        return before - torch.cuda.mem_get_info()[0], ctx.stats()


def test_second_pair_of_bit_rows_only_for_slices():
    """A dense closure of 9,216 constants takes one pair of bit rows (21 MB); a second one when a slice is tried, and none is
    tried where that does not fit."""
    n = 9216
    R = torch.ones((n, n), dtype=torch.uint8, device="cuda")
    R[:, 1500] = 0
    R[n - 100:, 1500] = 1
    out = torch.zeros_like(R)
    one, st = workspace_of(R, n, out, variant="rms_tc")  # one product fills the column
    assert int(out.min()) == 1 and st["e2m1_products"] == 1
    R[:801, n - 100:] = 0
    two, st = workspace_of(R, n, out, variant="rms_tc")  # a product, and a slice
    assert int(out.min()) == 1 and st["e2m1_products"] == 1 and st["thin_squarings"] == 2
    pair = 2 * n * (n // 64) * 8
    assert two - one > 0.9 * pair
    held = hold_all_but(one + pair // 2 + (6 << 20))
    try:
        some, st = workspace_of(R, n, out, variant="rms_tc")
        assert int(out.min()) == 1 and st["e2m1_products"] == 2
        assert some < two - pair // 2
    finally:
        del held
        torch.cuda.empty_cache()


def test_insertion_without_room_for_a_chunk():
    n = 131072  # 17 MB of scratch
    P = torch.zeros((n, wl.words(n)), dtype=torch.int64, device="cuda")
    facts = np.array([[1, 2], [5, 6], [3, 4], [9, 8], [7, 0], [2, 100000], [100000, 3]], np.int32)
    with pkg.Context(0) as ctx:
        want = P.clone()
        for f in facts:
            ctx.insert(want, n, f[None], fmt=PACKED)
        held = hold_all_but(8 << 20)
        try:
            ctx.insert(P, n, facts, fmt=PACKED)
            assert ctx.stats()["launches"] == len(facts)
            torch.cuda.synchronize()
        finally:
            del held
            torch.cuda.empty_cache()
        assert torch.equal(P, want) and bool(P[1, 0] & 0x1C == 0x1C)


def test_packed_composition_without_room_for_a_second_index():
    n = 9001
    a, b = wl.er_graph(n, 2.0, 5), wl.er_graph(n, 0.8, 6)
    A, B = (torch.from_numpy(wl.csr_to_packed(n, *x).view(np.int64)).cuda() for x in (a, b))
    out, again = torch.zeros_like(A), torch.zeros_like(A)
    torch.cuda.synchronize()
    with pkg.Context(0) as ctx:
        before = torch.cuda.mem_get_info()[0]
        ctx.compose(A, B, n, out, fmt=PACKED, variant="rms_packed")
        torch.cuda.synchronize()
        used = before - torch.cuda.mem_get_info()[0]
        launches = ctx.stats()["launches"]
    held = hold_all_but(used - n * (n // 64) * 8 // 2)
    try:
        with pkg.Context(0) as ctx:
            ctx.compose(A, B, n, again, fmt=PACKED, variant="rms_packed")
            torch.cuda.synchronize()
            assert ctx.stats()["launches"] < launches  # no index of R1 and no pass over its cost
    finally:
        del held
        torch.cuda.empty_cache()
    assert torch.equal(out, again)
    rows = np.arange(0, n, 97, dtype=np.int32)
    np.testing.assert_array_equal(wl.unpack_rows(out.cpu().numpy().view(np.uint64), n)[rows], oracle.compose_rows(n, a, b, rows))
