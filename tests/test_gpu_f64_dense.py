"""FP64 solves, whose rounds read kernel values formed once, against K from numpy: edges of the
32-row blocks and of the cluster's parts, the largest size that keeps the values and the first
that does not, every padded width, and column counts around the eight of a CTA and the 32 of a
launch.

Tolerance: the solves run until their residual's norm is below 1e-10; rounding adds at most about
2^-53 n per round to a row of K x (|x| <= 1, k_ij <= 1.4), 1e-9 for a hundred rounds at the largest
size.  2e-9 covers both."""
import numpy as np
import pytest
import torch

from paper_1501_05427_gb300 import ulisse as u

pytestmark = pytest.mark.gpu


def _check(n, d, R, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, d)).astype(np.float32)
    psi = np.concatenate([rng.uniform(-0.5, 0.0, d), [0.3, np.log(2.0)]])
    B = rng.choice([-1.0, 1.0], (n, R)).astype(np.float32)
    cfg = u.ulisse_config_default(precision=u.PREC_FP64, q=0.0, eps=1e-10, max_iter=2000)
    with u.Context(torch.from_numpy(X).cuda(), torch.zeros(n, device="cuda"), cfg) as ctx:
        S, _ = ctx.solve(psi, torch.from_numpy(B).cuda(), n_est=np.ones(R, dtype=np.int32), step=1)
    S = S.cpu().numpy().astype(np.float64)
    Z = X.astype(np.float64) * np.exp(-psi[:d])
    sq = (Z * Z).sum(1)
    K = np.exp(psi[d] - 0.5 * np.maximum(sq[:, None] + sq[None, :] - 2.0 * Z @ Z.T, 0.0))
    K[np.diag_indices(n)] += np.exp(psi[d + 1])
    # S comes back in 32 bits: its rounding passes through K
    tol = 2e-9 + 2.0 ** -24 * (np.abs(K) @ np.abs(S))
    assert np.all(np.abs(K @ S - B) <= tol)


@pytest.mark.parametrize("n", [1, 7, 31, 33, 257, 1000, 2049, 5792, 5793])
def test_sizes(n):
    _check(n, 3, 3, n)


@pytest.mark.parametrize("d,R", [(1, 1), (2, 7), (4, 8), (5, 9), (8, 17), (11, 32), (16, 33)])
def test_widths(d, R):
    _check(300, d, R, d)
