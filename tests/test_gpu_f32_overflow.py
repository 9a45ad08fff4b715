"""FP32 products at the largest sigma^2: kernel values beyond the largest BF16 value keep their FP32
result, and infinite ones make a positive sum an infinity, not a NaN (but the derivative's own term,
k_ii times zero, is NaN then, and every row has one).

V > 0.  Every row is infinite when k_ii = sigma^2 is beyond the largest float by more than the kernel
value's own error (FP32 exponents of 128: 2e-5), and finite where its sum is below the largest
float.  (The SIMT kernel multiplies the padding of its last 64-point tile too, an infinite value
times zero near the origin, so it is no reference for the pattern; its finite entries agree within
the FP32 products' stated bound of 1e-5.)"""
import numpy as np
import pytest
import torch

from paper_1501_05427_gb300 import ulisse as u

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [300, 3001])
@pytest.mark.parametrize("which", [-1, 0, 2])
@pytest.mark.parametrize("log_sigma2", [88.0, 88.722, 88.8, 89.0, 100.0])
def test_largest_sigma2(n, which, log_sigma2):
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 2)).astype(np.float32)
    V = torch.from_numpy(rng.uniform(1e-6, 1e-3, (n, 9)).astype(np.float32)).cuda()
    psi = np.array([-0.5, 0.1, log_sigma2, -1.0])
    U = []
    for rows in (0, 2):
        cfg = u.ulisse_config_default(kmv_rows_per_thread=rows)
        with u.Context(torch.from_numpy(X).cuda(), torch.zeros(n, device="cuda"), cfg) as ctx:
            U.append(ctx.kmv(psi, V, which=which).cpu().numpy())
    a, b = U
    Z = X.astype(np.float64) * np.exp(-psi[:2])
    kmax = np.exp(psi[2])     # k_ii, the row's largest
    big = float(np.finfo(np.float32).max)
    if which == 0:
        assert np.all(np.isnan(a)) if kmax > big * (1 + 2e-5) else np.all(np.isfinite(a))
    elif kmax > big * (1 + 2e-5):
        assert np.all(a == np.inf)
    else:
        exact = np.exp(psi[2] - 0.5 * ((Z[:, None] - Z[None]) ** 2).sum(2)) @ V.cpu().numpy().astype(float)
        exact += np.exp(psi[3]) * V.cpu().numpy() if which == -1 else 0.0
        assert np.all(a > 0)   # a sum may overflow, to an infinity
        assert np.all(np.isfinite(a[exact < (1 - 1e-4) * big]))
    both = np.isfinite(a) & np.isfinite(b)
    assert np.all(np.abs(a[both].astype(np.float64) - b[both]) <= 1e-5 * np.abs(b[both]))
