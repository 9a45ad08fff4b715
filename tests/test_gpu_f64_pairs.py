"""FP64 products over unordered block pairs (K V and its derivatives at n where the pair form
applies) against the oracle: edges of the 32- and 64-point blocks, the size where the block
changes (2,048), every padded width, one to 40 columns, and kernel values from 1 down to
underflow (far points take the exponential's library branch).

Tolerance: the products' relative error per entry of Sum_j |A_ij| |V_jr| is bounded by a few
units of 2^-53 per distance dimension, per term and for the exponential; 1e-12, as the other
FP64 parity tests, covers n <= 2,500 terms with a factor over 100 to spare."""
import numpy as np
import pytest
import torch

import oracle
from paper_1501_05427_gb300 import ulisse as u

pytestmark = pytest.mark.gpu


def _check(n, d, R, which, spread, seed):
    rng = np.random.default_rng(seed)
    X = (rng.standard_normal((n, d)) * spread).astype(np.float32)
    psi = np.concatenate([rng.uniform(-0.5, 0.5, d), [0.3, np.log(0.2)]])
    V = rng.standard_normal((n, R))
    rows = np.unique(np.concatenate([[0, n - 1], rng.integers(0, n, 60)]))
    ctx = u.Context(torch.from_numpy(X).cuda(), torch.zeros(n, device="cuda"),
                    u.ulisse_config_default(precision=u.PREC_FP64))
    with ctx:
        U = ctx.kmv(psi, torch.from_numpy(V).cuda(), which=which).cpu().numpy()
    Xd = X.astype(np.float64)
    if which == -1:
        ref = oracle.kmv_rows(Xd, psi, V, rows)
        scale = oracle.kmv_rows(Xd, psi, V, rows, absolute=True)
    else:
        ref = oracle.kmv(Xd, psi, V, which)[rows]
        scale = oracle.kmv(Xd, psi, np.abs(V), which)[rows]
    err = np.abs(U[rows] - ref)
    assert np.all(err <= 1e-12 * scale + 1e-300), (np.max(err / np.maximum(scale, 1e-300)))


@pytest.mark.parametrize("n", [1, 31, 32, 33, 65, 1000, 2048, 2049, 2500])
def test_pair_edges(n):
    _check(n, 2, 5, -1, 0.5, n)


@pytest.mark.parametrize("d,R", [(1, 1), (3, 32), (5, 33), (8, 40), (16, 2)])
def test_pair_widths(d, R):
    _check(193, d, R, -1, 1.0, 10 * d + R)


@pytest.mark.parametrize("which", [0, 2, 3])
def test_pair_derivatives(which):
    _check(301, 3, 3, which, 0.7, which)


def test_pair_far_points():
    # distances from 0 to tens of thousands: kernel values through the whole normal range, the
    # denormals and zero
    _check(400, 2, 3, -1, 40.0, 7)
