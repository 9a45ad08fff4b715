"""After a bounded wait that ran out, a batch is usable again: the counters by which a launch finds
its last CTA are zeroed, the batch's and its problems'.

The self-test leaves counts in them that no launch completes, so that a counter that was not zeroed
shows as a product or a gradient that is never written.  The outputs are sums in a fixed order,
hence equal bit for bit."""
import numpy as np
import pytest
import torch

from paper_1501_05427_gb300 import ulisse as u
from paper_1501_05427_gb300 import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [u.PREC_FP32, u.PREC_MIXED])
def test_batch_after_timeout(precision):
    probs = [w.census_like(n=n, seed=n) for n in (300, 1030, 9_001)]
    Xs = [torch.from_numpy(p.X).cuda() for p in probs]
    ys = [torch.from_numpy(p.y).cuda() for p in probs]
    psi = np.concatenate([p.psi_true for p in probs])
    Vs = [torch.randn(9, p.n, device="cuda").t() for p in probs]
    with u.BatchContext(Xs, ys, u.ulisse_config_default(precision=precision, seed=2)) as ctx:
        U0 = [U.clone() for U in ctx.kmv(psi, Vs)]
        g0, _ = ctx.grad(psi, step=3)
        assert ctx._lib.ulisse_selftest_wait_timeout(ctx._h) == u.ULISSE_ERR_TIMEOUT
        for U, ref in zip(ctx.kmv(psi, Vs), U0):
            assert torch.equal(U, ref)
        assert ctx._lib.ulisse_selftest_wait_timeout(ctx._h) == u.ULISSE_ERR_TIMEOUT
        g, _ = ctx.grad(psi, step=3)
    assert np.array_equal(g, g0)
