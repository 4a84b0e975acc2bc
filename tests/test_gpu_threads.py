"""Calls of several host threads with a context each, on kernels whose shared memory depends on the size: the largest launch
is not refused because a smaller one comes between its preparation and its launch. (Several threads with small calls, since
the time between the two is about a microsecond.)"""
import threading

import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pkg = pytest.importorskip("paper_2408_10369_gb300")

pytestmark = pytest.mark.gpu
PACKED = pkg.BMLP_FMT_PACKED64


def closure_call(n, d, variant):
    ip, ix = wl.er_graph(n, d, n)
    R = torch.from_numpy(wl.csr_to_packed(n, ip, ix).view(np.int64)).cuda()
    out = torch.zeros_like(R)
    return lambda ctx, s: ctx.rms(R, n, out, fmt=PACKED, variant=variant, stream=s), out, wl.pack_rows(oracle.closure(n, ip, ix))


def query_call(n, d, q, variant="auto"):
    ip, ix = wl.er_graph(n, d, n)
    R = torch.from_numpy(wl.csr_to_packed(n, ip, ix).view(np.int64)).cuda()
    src = wl.query_rows(n, q, 1, 4, 7)
    dev, out = torch.from_numpy(src.view(np.int64)).cuda(), torch.zeros((q, wl.words(n)), dtype=torch.int64, device="cuda")
    return lambda ctx, s: ctx.smp(R, n, dev, q, out, fmt=PACKED, variant=variant, stream=s), out, wl.pack_rows(oracle.smp(n, ip, ix, src)[0])


@pytest.mark.parametrize("kind", ["small", "query", "tiles", "rows"])
def test_threads(kind):
    small, large, calls = {
        "small": (lambda k: closure_call(60 + k, 2.0, "auto"), lambda: closure_call(1000, 2.0, "auto"), 3000),
        "query": (lambda k: query_call(500 + k, 0.5, 1), lambda: query_call(100000, 0.3, 1), 3000),
        "tiles": (lambda k: query_call(4096 + k, 4.0, 64), lambda: query_call(16000, 4.0, 64), 800),
        "rows": (lambda k: closure_call(100 + k, 1.0, "smp_packed"), lambda: query_call(20000, 0.3, 64), 2000)}[kind]
    work = [small(k) for k in range(5)] + [large()]
    errors = []
    start = threading.Barrier(len(work))
    done = threading.Event()

    def run(call, last):
        ctx = pkg.Context(0)
        try:
            stream = torch.cuda.Stream()
            call(ctx, stream)
            start.wait()
            for _ in range(calls):
                call(ctx, stream)
                if done.is_set():
                    break
            stream.synchronize()
        except Exception as e:  # noqa: BLE001
            errors.append(e)
            start.abort()
        finally:
            if last:
                done.set()
            ctx.close()

    threads = [threading.Thread(target=run, args=(c, k == len(work) - 1)) for k, (c, _, _) in enumerate(work)]
    torch.cuda.synchronize()
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for _, out, want in work:
        np.testing.assert_array_equal(out.cpu().numpy().view(np.uint64), want)
