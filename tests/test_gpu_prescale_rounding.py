"""x / l in FP32 is the FP64 product x (1 / l) rounded to 32 bits, also for the inputs within 2^-47 of the
middle between two floats, which a product with 1 / l as a pair of floats rounds the other way.

Bit for bit: products on the inputs with their lengthscale against products on inputs that numpy has
scaled, with lengthscale one."""
import numpy as np
import pytest
import torch

from paper_1501_05427_gb300 import ulisse as u

pytestmark = pytest.mark.gpu

# log l and an x whose two roundings differ (found over all x in [1, 2)); 1 / l may be off by a unit
# in its last place without a change
NEAR = [(0.09, "0x1.fa781cp+0"), (0.15, "0x1.e1f72p+0"), (0.19, "0x1.98d01ep+0"),
        (0.31, "0x1.3565f4p+0"), (0.35, "0x1.60ddb8p+0"), (0.43, "0x1.70eb12p+0")]


def _kmv(X, psi, V, which, precision):
    cfg = u.ulisse_config_default(precision=precision)
    with u.Context(torch.from_numpy(X).cuda(), torch.zeros(len(X), device="cuda"), cfg) as ctx:
        return ctx.kmv(psi, V, which=which)


@pytest.mark.parametrize("precision", [u.PREC_FP32, u.PREC_MIXED])
@pytest.mark.parametrize("log_l,x", NEAR)
def test_nearly_halfway(precision, log_l, x):
    # the x at several powers of two and both signs, among ordinary inputs
    x = np.float32(float.fromhex(x))
    X = np.concatenate([x * np.float32(2.0) ** np.arange(-3, 2), -x * np.float32(2.0) ** np.arange(-3, 2),
                        np.linspace(-2, 2, 53)]).astype(np.float32)[:, None]
    Xs = (X.astype(np.float64) * np.exp(-log_l)).astype(np.float32)
    V = torch.from_numpy(np.random.default_rng(1).standard_normal((len(X), 6)).astype(np.float32)).cuda()
    for which in (-1, 0):
        a = _kmv(X, np.array([log_l, 0.1, -1.0]), V, which, precision)
        b = _kmv(Xs, np.array([0.0, 0.1, -1.0]), V, which, precision)
        assert torch.equal(a, b)
