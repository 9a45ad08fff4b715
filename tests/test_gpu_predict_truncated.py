"""FP64 predictions with q > 0 are made from the truncated estimates of ulisse_solve, rounding
included: over the fifty and more CG rounds of an ill-conditioned problem another exponential or
another order of additions gives another trajectory, hence another estimate.

The mean at m test inputs comes from one column, y, as a solve of y alone does.  Tolerance: that
solve returns its estimate s in 32 bits and the mean comes back in 32 bits, 2^-24 of
Sum_i k*_ij |s_i| and of the mean; the FP64 sums' rounding is far below.  (In numpy, kernel values
off by 2^-52 move these means by 20 to 6,000 times that.)"""
import numpy as np
import pytest
import torch

from paper_1501_05427_gb300 import ulisse as u

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ls,noise,q", [(300, 0.3, 1e-3, 0.1), (600, 0.1, 1e-3, 0.02),
                                          (1000, 0.3, 1e-6, 0.1)])
def test_mean_is_the_solves(n, ls, noise, q):
    rng = np.random.default_rng(n)
    X = rng.uniform(0, 1, (n, 2)).astype(np.float32)
    y = rng.choice([-1.0, 1.0], n).astype(np.float32)
    psi = np.array([np.log(ls), np.log(ls), 0.0, np.log(noise)])
    Xs = rng.uniform(-0.5, 1.5, (64, 2)).astype(np.float32)
    cfg = u.ulisse_config_default(precision=u.PREC_FP64, q=q, max_iter=20000, seed=5)
    yd = torch.from_numpy(y).cuda()
    with u.Context(torch.from_numpy(X).cuda(), yd, cfg) as ctx:
        S, stats = ctx.solve(psi, yd[:, None], step=7)
        mean, _ = ctx.predict(psi, torch.from_numpy(Xs).cuda(), step=7, var=False)
    assert stats[0][1] >= 50     # rounds: enough for the rounding to matter
    mean = mean.cpu().numpy().astype(np.float64)
    s = S[:, 0].cpu().numpy().astype(np.float64)
    Z, Zs = X.astype(np.float64) / ls, Xs.astype(np.float64) / ls
    k = np.exp(-0.5 * ((Zs[:, None, :] - Z[None, :, :]) ** 2).sum(2))
    ref = k @ s
    tol = 1.01 * 2.0 ** -24 * (k @ np.abs(s) + np.abs(ref))
    assert np.all(np.abs(mean - ref) <= tol), np.max(np.abs(mean - ref) / tol)
