"""The bound of the in-kernel waits is that of the call, also for a batch whose graph is kept: the same batch on one context
with a bound of one nanosecond, which no pipeline can meet, and with the default, in both orders."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pkg = pytest.importorskip("paper_2408_10369_gb300")
from paper_2408_10369_gb300 import bmlp  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1500, 4500])  # grouped, and a pipeline of its own
def test_batch_timeout_follows_the_call(n):
    csr = wl.er_graph(n, n / 5, 3)  # dense: on the tensor cores
    R = torch.from_numpy(wl.dense_u8(n, *csr)).cuda()
    out = torch.zeros_like(R)
    items = pkg.Context.problems([dict(n=n, R1=R, out=out)])
    want = oracle.closure(n, *csr)
    with pkg.Context(0) as ctx:
        for _ in range(2):
            with pytest.raises(bmlp.BmlpError) as e:
                ctx.batch_run(items, timeout_ns=1)
            assert e.value.status == bmlp.BMLP_ERR_TIMEOUT
            out.zero_()
            ctx.batch_run(items)
            torch.cuda.synchronize()
            np.testing.assert_array_equal(out.cpu().numpy(), want)
