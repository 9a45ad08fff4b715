"""A product whose results are NaN takes about as long as any other: a NaN among the inputs (every
kernel value of that point), or an infinity in a column of V, which leaves one column to be formed
again from its terms that are not finite.

Bound: twice the time of the same product with finite results, medians of 9 calls (the columns'
words are one pass over 4 bytes per 32 points and column)."""
import numpy as np
import pytest
import torch

from paper_1501_05427_gb300 import ulisse as u

pytestmark = pytest.mark.gpu


def _time(ctx, psi, V, U):
    t = []
    for _ in range(12):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        ctx.kmv(psi, V, out=U)
        b.record()
        b.synchronize()
        t.append(a.elapsed_time(b))
    return sorted(t[3:])[4]


@pytest.mark.parametrize("n,R", [(22_784, 17), (5_000, 32)])
def test_cost(n, R):
    g = torch.Generator("cuda").manual_seed(n)
    X = torch.randn(n, 8, generator=g, device="cuda")
    V = torch.randn(R, n, generator=g, device="cuda").t()
    U = torch.empty(R, n, device="cuda").t()
    psi = np.concatenate([np.zeros(9), [-2.0]])
    y = torch.zeros(n, device="cuda")
    with u.Context(X, y, u.ulisse_config_default()) as ctx:
        finite = _time(ctx, psi, V, U)
        W = V.t().clone().t()
        W[7, 3] = float("inf")
        inf_v = _time(ctx, psi, W, U)
        assert torch.all(U[:, 3] == float("inf")) and torch.all(torch.isfinite(U[:, :3]))
    X[11, 2] = float("nan")
    with u.Context(X, y, u.ulisse_config_default()) as ctx:
        nan_x = _time(ctx, psi, V, U)
        assert torch.all(torch.isnan(U))
    print("n=%d R=%d: finite %.3f ms, an infinity in V %.3f ms, a NaN in X %.3f ms"
          % (n, R, finite, inf_v, nan_x))
    assert inf_v <= 2 * finite and nan_x <= 2 * finite
