"""FP32 batches on the tensor cores (five columns and more): a batch takes that form at every size,
and a CTA several ranges of a problem's split where many problems fill the SMs; a problem's product
is the one it has alone, bit for bit, whatever the batch (sizes of up to 10,000 points, where a
context of its own takes the same form), and within the FP32 products' bound of 1e-5 of the oracle
above."""
import numpy as np
import pytest
import torch

import oracle
from paper_1501_05427_gb300 import ulisse as u

pytestmark = pytest.mark.gpu


def _problem(n, d, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, d)).astype(np.float32)
    return X, np.concatenate([rng.uniform(-0.4, 0.6, d), [0.2, np.log(0.1)]])


# few problems (a CTA per range), and enough to give a CTA 32 tiles: edges of the tiles, the row
# blocks and the ranges
SIZES = {"few": [255, 256, 1_030, 4_097],
         "many": [257, 288, 383, 500, 641, 1_023, 1_025, 1_500, 2_000, 3_001, 8_193, 9_999] * 6}


@pytest.mark.parametrize("R", [5, 9, 17, 32])
@pytest.mark.parametrize("kind", ["few", "many"])
def test_same_as_alone(kind, R):
    ns = SIZES[kind]
    probs = [_problem(n, (1, 2, 4, 8)[b % 4], b) for b, n in enumerate(ns)]
    Xs = [torch.from_numpy(X).cuda() for X, _ in probs]
    ys = [torch.zeros(n, device="cuda") for n in ns]
    Vs = [torch.randn(R, n, device="cuda", generator=torch.Generator("cuda").manual_seed(n)).t() for n in ns]
    with u.BatchContext(Xs, ys, u.ulisse_config_default()) as ctx:
        Us = ctx.kmv(np.concatenate([p for _, p in probs]), Vs)
    for b in range(min(len(ns), 12)):
        with u.Context(Xs[b], ys[b], u.ulisse_config_default()) as ctx:
            U = ctx.kmv(probs[b][1], Vs[b])
        if ns[b] >= 256:
            assert torch.equal(U, Us[b]), ns[b]
        else:     # the SIMT kernels of a batch and of a context add in other orders
            assert torch.linalg.norm(U - Us[b]) <= 1e-5 * torch.linalg.norm(U)


@pytest.mark.parametrize("R", [5, 6, 9])
def test_large_problems(R):
    ns = [12_000, 700, 20_011]
    probs = [_problem(n, 8, n) for n in ns]
    Vs = [np.random.default_rng(n).standard_normal((n, R)).astype(np.float32) for n in ns]
    with u.BatchContext([torch.from_numpy(X).cuda() for X, _ in probs],
                        [torch.zeros(n, device="cuda") for n in ns], u.ulisse_config_default()) as ctx:
        Us = ctx.kmv(np.concatenate([p for _, p in probs]), [torch.from_numpy(V).cuda() for V in Vs])
    for (X, psi), V, U in zip(probs, Vs, Us):
        rows = np.unique(np.r_[0, len(X) - 1, np.random.default_rng(1).integers(0, len(X), 30)])
        Xd, Vd = X.astype(np.float64), V.astype(np.float64)
        ref = oracle.kmv_rows(Xd, psi, Vd, rows)
        scale = oracle.kmv_rows(Xd, psi, Vd, rows, absolute=True)
        assert np.max(np.abs(U.cpu().numpy()[rows] - ref) / scale) <= 1e-5


def test_not_slower_on_both_sides_of_a_size():
    # sizes around 10,000, where a context of its own changes its form at 5 and 6 columns: there as
    # at 7 columns (two launches with a tail each took 2.2 times as long)
    ns = [11_000, 9_000, 12_000, 5_000, 8_000, 11_500, 3_000, 9_900]
    probs = [_problem(n, 4, n) for n in ns]
    psi = np.concatenate([p for _, p in probs])
    ms = {}
    with u.BatchContext([torch.from_numpy(X).cuda() for X, _ in probs],
                        [torch.zeros(n, device="cuda") for n in ns], u.ulisse_config_default()) as ctx:
        for R in (5, 7):
            Vs = [torch.randn(R, n, device="cuda").t() for n in ns]
            t = []
            for _ in range(14):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                ctx.kmv(psi, Vs)
                b.record()
                b.synchronize()
                t.append(a.elapsed_time(b))
            ms[R] = sorted(t[4:])[5]
    print("5 columns %.3f ms, 7 columns %.3f ms" % (ms[5], ms[7]))
    assert ms[5] <= 1.2 * ms[7]
