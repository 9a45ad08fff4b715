"""Gradients after a call that grows the context's column buffers: the columns' metadata (estimator
counts and offsets) goes with the buffers and is made again.  Bit for bit the gradient before the
growth, and a fresh context's."""
import numpy as np
import pytest
import torch

from paper_1501_05427_gb300 import ulisse as u
from paper_1501_05427_gb300 import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [u.PREC_FP32, u.PREC_MIXED, u.PREC_FP64])
@pytest.mark.parametrize("by", ["kmv", "predict", "bilinear"])
def test_gradient_after_growth(precision, by):
    prob = w.census_like(n=700, seed=12)
    X, y = torch.from_numpy(prob.X).cuda(), torch.from_numpy(prob.y).cuda()
    cfg = u.ulisse_config_default(precision=precision, seed=4)
    V = torch.randn(40, prob.n, device="cuda").t()
    with u.Context(X, y, cfg) as ctx:
        g0, st0 = ctx.grad(prob.psi_true, step=3)
        if by == "kmv":
            ctx.kmv(prob.psi_true, V)
        elif by == "predict":
            ctx.predict(prob.psi_true, X[:20].contiguous(), step=1)
        else:
            ctx.dk_bilinear(prob.psi_true, V, V)
        g1, st1 = ctx.grad(prob.psi_true, step=3)
    with u.Context(X, y, cfg) as ctx:
        ref, st = ctx.grad(prob.psi_true, step=3)
    assert st0 == st1 == st
    assert np.array_equal(g0, ref) and np.array_equal(g1, ref)
