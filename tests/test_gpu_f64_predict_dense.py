"""FP64 predictions to convergence (q = 0), whose solves read kernel values formed once by the
table-driven exponential with sums in any order (solves through ulisse_solve, and the file
test_gpu_f64_dense.py with them, take the ordered form), against a dense solve in 64 bits: edges of the
32-row blocks and of the cluster's eight parts, empty parts (n < 8), the largest size that keeps the
values and the first that does not, every padded width, and column counts giving a CTA each width
from one to eight, one launch of more than 32 columns, and the mean alone.

Tolerance: the solves stop at residuals of 1e-10 and lambda = 2, so their error times |k*| is below
1e-8; the outputs come back in 32 bits, 2^-24 of the mean and of sigma^2 + lambda."""
import numpy as np
import pytest
import torch

from paper_1501_05427_gb300 import ulisse as u

pytestmark = pytest.mark.gpu


def _check(n, d, m, var=True):
    g = torch.Generator("cuda").manual_seed(1000 * n + 10 * d + m)
    X = torch.rand(n, d, generator=g, device="cuda")
    y = torch.randn(n, generator=g, device="cuda")
    Xs = torch.rand(m, d, generator=g, device="cuda")
    psi = np.concatenate([np.linspace(-1.0, 0.2, d), [0.3, np.log(2.0)]])
    cfg = u.ulisse_config_default(precision=u.PREC_FP64, q=0.0, eps=1e-10, max_iter=3000)
    with u.Context(X, y, cfg) as ctx:
        mean, v = ctx.predict(psi, Xs, var=var)
    inv = torch.from_numpy(np.exp(-psi[:d])).cuda()
    Z, Zs = X.double() * inv, Xs.double() * inv
    dist = lambda a, b: torch.cdist(a, b, compute_mode="donot_use_mm_for_euclid_dist") ** 2
    s2, lam = np.exp(psi[d]), np.exp(psi[d + 1])
    K = s2 * torch.exp(-0.5 * dist(Z, Z))
    K.diagonal().add_(lam)
    ks = s2 * torch.exp(-0.5 * dist(Z, Zs))
    S = torch.linalg.solve(K, torch.cat([y.double()[:, None], ks], 1))
    mean_ref, var_ref = ks.t() @ S[:, 0], s2 + lam - (ks * S[:, 1:]).sum(0)
    assert torch.all((mean - mean_ref).abs() <= 2.0 ** -23 * mean_ref.abs() + 1e-8)
    if var:
        assert torch.all((v - var_ref).abs() <= 2.0 ** -23 * (s2 + lam) + 1e-8)


@pytest.mark.parametrize("n", [1, 7, 31, 33, 257, 1030, 2049, 5791, 5792, 5793])
def test_sizes(n):
    _check(n, 2, 4)


@pytest.mark.parametrize("d", [1, 3, 8, 16])
def test_widths(d):
    _check(331, d, 6)


@pytest.mark.parametrize("columns", [1, 2, 3, 4, 5, 6, 7, 8, 9, 13, 32, 33, 101, 300])
def test_columns(columns):
    _check(203, 2, max(1, columns - 1), var=columns > 1)
