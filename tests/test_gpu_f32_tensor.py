"""FP32 products with the contraction on the tensor cores against the oracle: edges of the 32-point
tiles, 128-row blocks and split ranges, every padded width, column counts around the two MMA
widths and the 32-column launches, derivatives, and the same products by the SIMT kernel
(kmv_rows_per_thread fixes that form).

Tolerance, per entry relative to Sum_j |A_ij| |V_jr|: the kernel value's own error (the prescaled
inputs' rounding and ex2, about 1e-6 at these distances) plus 2^-22 for the products left out of
the split, the truncating tile sums and n / 32 FP32 additions of at most 2^-24 each: below 1e-5,
the FP32 products' stated bound."""
import numpy as np
import pytest
import torch

import oracle
from paper_1501_05427_gb300 import ulisse as u

pytestmark = pytest.mark.gpu


def _problem(n, d, R, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, d)).astype(np.float32)
    psi = np.concatenate([rng.uniform(-0.4, 0.6, d), [0.2, np.log(0.1)]])
    V = rng.standard_normal((n, R)).astype(np.float32)
    rows = np.unique(np.concatenate([[0, n - 1, n // 2], rng.integers(0, n, 40)]))
    return X, psi, V, rows


def _run(X, psi, V, which=-1, rows_per_thread=0):
    cfg = u.ulisse_config_default(kmv_rows_per_thread=rows_per_thread)
    with u.Context(torch.from_numpy(X).cuda(), torch.zeros(len(X), device="cuda"), cfg) as ctx:
        return ctx.kmv(psi, torch.from_numpy(V).cuda(), which=which).cpu().numpy()


def _check(n, d, R, which=-1):
    X, psi, V, rows = _problem(n, d, R, 7 * n + R)
    U = _run(X, psi, V, which)[rows]
    Xd, Vd = X.astype(np.float64), V.astype(np.float64)
    if which == -1:
        ref = oracle.kmv_rows(Xd, psi, Vd, rows)
        scale = oracle.kmv_rows(Xd, psi, Vd, rows, absolute=True)
    else:
        ref = oracle.kmv(Xd, psi, Vd, which)[rows]
        scale = oracle.kmv(Xd, psi, np.abs(Vd), which)[rows]
    assert np.max(np.abs(U - ref) / scale) <= 1e-5


@pytest.mark.parametrize("n", [255, 256, 257, 288, 383, 385, 1030, 4097, 20011])
def test_sizes(n):
    _check(n, 8, 9)


@pytest.mark.parametrize("R", [5, 7, 15, 16, 17, 31, 32, 33, 37, 70])
def test_columns(R):
    _check(641, 4, R)


@pytest.mark.parametrize("d", [1, 2, 3, 5, 8, 11, 16])
def test_widths(d):
    _check(517, d, 6)


@pytest.mark.parametrize("which", [0, 2, 3, 4])
def test_derivatives(which):
    _check(421, 3, 8, which)


def test_same_as_simt():
    X, psi, V, _ = _problem(3001, 8, 17, 3)
    a, b = _run(X, psi, V), _run(X, psi, V, rows_per_thread=2)
    assert np.linalg.norm(a - b) <= 2e-6 * np.linalg.norm(b)


def test_not_finite():
    # a column that holds an infinity or a NaN leaves the others alone
    X, psi, V, _ = _problem(700, 2, 6, 5)
    U0 = _run(X, psi, V)
    W = V.copy()
    W[10, 1], W[20, 4] = np.inf, np.nan
    U = _run(X, psi, W)
    keep = [0, 2, 3, 5]
    assert np.array_equal(U[:, keep], U0[:, keep])
    assert not np.isfinite(U[10, 1]) and np.all(np.isnan(U[:, 4]))


@pytest.mark.parametrize("n", [300, 700, 5001])
@pytest.mark.parametrize("which", [-1, 1])
def test_infinities(n, which):
    # k_ij > 0 at these distances: one infinity is every row's, both signs are NaN, and the
    # SIMT kernel says the same (the derivative's k_jj is 0: NaN in the infinity's own row)
    X, psi, V, _ = _problem(n, 2, 6, 11)
    V[5, 0], V[n - 1, 2], V[7, 3], V[n - 2, 3], V[9, 4] = np.inf, -np.inf, np.inf, -np.inf, np.nan
    a, b = _run(X, psi, V, which), _run(X, psi, V, which, rows_per_thread=2)
    bad = [0, 2, 3, 4]
    assert np.array_equal(a[:, bad], b[:, bad], equal_nan=True)
    assert np.all(np.isfinite(a[:, [1, 5]]))
    if which == -1:
        assert np.all(a[:, 0] == np.inf) and np.all(a[:, 2] == -np.inf)
        assert np.all(np.isnan(a[:, 3])) and np.all(np.isnan(a[:, 4]))


def test_largest_floats():
    # the largest floats are beyond the largest BF16 value, and finite times k_ij < 1
    X, psi, V, rows = _problem(700, 2, 6, 13)
    psi[2] = -1.0
    V[10, 1], V[20, 4] = np.finfo(np.float32).max, -np.finfo(np.float32).max
    U = _run(X, psi, V)[rows]
    Xd, Vd = X.astype(np.float64), V.astype(np.float64)
    ref = oracle.kmv_rows(Xd, psi, Vd, rows)
    scale = oracle.kmv_rows(Xd, psi, Vd, rows, absolute=True)
    assert np.max(np.abs(U - ref) / scale) <= 1e-5
