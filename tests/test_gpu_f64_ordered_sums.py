"""Truncated FP64 solves keep one order of additions at every size, also where a column's sums span
more chunks of 2,048 rows than a cluster has CTAs (n > 16,384).

A problem gets points with a zero right-hand side so far away that their kernel values are zero:
they add chunks of zeros at the end of every sum and, at the sizes taken on 152 SMs, leave the
products' split ranges as they are, so that the solve of the other points is the same arithmetic
with 9, 13 and 16 chunks.  Over the hundred and more rounds of an ill-conditioned problem any
other order of additions gives another estimate (here 1e-3 off); the estimates come back equal bit
for bit."""
import math

import numpy as np
import pytest
import torch

from paper_1501_05427_gb300 import ulisse as u

pytestmark = pytest.mark.gpu

N = 16_384


def _solve(extra):
    rng = np.random.default_rng(4)
    X = np.concatenate([rng.uniform(0, 1, (N, 2)), np.full((extra, 2), 1e3)]).astype(np.float32)
    b = np.concatenate([rng.choice([-1.0, 1.0], N), np.zeros(extra)]).astype(np.float32)
    psi = np.array([np.log(0.1), np.log(0.1), 0.0, np.log(0.05)])
    cfg = u.ulisse_config_default(precision=u.PREC_FP64, q=0.05 * math.sqrt(N / (N + extra)),
                                  max_iter=2000, seed=5)
    with u.Context(torch.from_numpy(X).cuda(), torch.zeros(N + extra, device="cuda"), cfg) as ctx:
        S, stats = ctx.solve(psi, torch.from_numpy(b).cuda()[:, None], step=7)
    assert not S[N:].any()
    return S[:N, 0].cpu().numpy(), stats[0][:3]


@pytest.mark.parametrize("extra", [10_240, 16_384])
def test_more_chunks(extra):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the sizes keep the split ranges on 152 SMs")
    ref, st_ref = _solve(2_048)
    S, st = _solve(extra)
    assert st_ref[1] >= 100 and st == st_ref
    assert np.array_equal(S, ref)
