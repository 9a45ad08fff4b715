"""FP32 tensor-core products where one term makes a row (lengthscales far below the points' distances,
K = sigma^2 I): no chain of additions hides the contraction's own rounding.

Bound per entry, of |K_ii v_i|: a tile's product is truncated at 12 accumulations, two of the product's
own size, 2.1 2^-23; the products left out of the split are below 2^-25; lambda v rounds once, 2^-24
of the sum (1 + lambda).  sigma^2 = 1, so that k_ii is exact."""
import numpy as np
import pytest
import torch

from paper_1501_05427_gb300 import ulisse as u

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [256, 1030, 5000])
@pytest.mark.parametrize("d", [1, 4, 16])
def test_one_term_rows(n, d):
    g = torch.Generator("cuda").manual_seed(n + d)
    X = torch.randn(n, d, generator=g, device="cuda")
    X[:, 0] = torch.arange(n, device="cuda")      # at least 100 lengthscales apart
    V = torch.randn(9, n, generator=g, device="cuda").t()
    lam = 0.05
    psi = np.concatenate([np.full(d, np.log(0.01)), [0.0, np.log(lam)]])
    with u.Context(X, torch.zeros(n, device="cuda"), u.ulisse_config_default()) as ctx:
        U = ctx.kmv(psi, V).double()
    ref = (1.0 + np.exp(np.log(lam))) * V.double()
    bound = (2.1 * 2.0 ** -23 + 2.0 ** -25 + (1 + lam) * 2.0 ** -23) * V.double().abs()
    assert torch.all((U - ref).abs() <= bound)
