"""FP64 calls without the memory for their scratch fall back on the row-block kernel: a product whose
pair form would take 256 MiB, and a solve whose formed kernel values would.

A tensor takes all of the device's memory but 128 MiB meanwhile.  The products agree within the FP64
parity bound, 1e-12 of Sum_j |K_ij| |V_jr| (K >= 0, V > 0: of the product itself); the truncated solves
keep one rounding, so they are equal bit for bit."""
import numpy as np
import pytest
import torch

from paper_1501_05427_gb300 import ulisse as u

pytestmark = pytest.mark.gpu


def _fill():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(free - (128 << 20), dtype=torch.uint8, device="cuda")


def _ctx(n, d, **cfg):
    g = torch.Generator("cuda").manual_seed(n)
    X = torch.rand(n, d, generator=g, device="cuda")
    c = u.ulisse_config_default(precision=u.PREC_FP64, seed=2, max_iter=3000, **cfg)
    return u.Context(X, torch.zeros(n, device="cuda"), c)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_product(dtype):
    n, R = 8_000, 32
    V = torch.rand(R, n, device="cuda", dtype=dtype).t()
    psi = np.array([-1.0, -1.2, 0.3, -2.0])
    with _ctx(n, 2) as ctx:
        U = torch.empty(R, n, device="cuda", dtype=dtype).t()
        filler = _fill()
        ctx.kmv(psi, V, out=U)
        torch.cuda.synchronize()
        del filler
        torch.cuda.empty_cache()
    with _ctx(n, 2) as ctx:
        ref = ctx.kmv(psi, V)
    tol = 1e-12 if dtype == torch.float64 else 2.0 ** -23
    assert torch.all((U - ref).abs() <= tol * ref)


@pytest.mark.parametrize("R", [1, 8, 9, 33])
def test_truncated_solve(R):
    n = 5_700
    B = torch.from_numpy(np.random.default_rng(R).choice([-1.0, 1.0], (n, R)).astype(np.float32)).cuda()
    psi = np.array([np.log(0.3), np.log(0.3), 0.0, np.log(0.05)])
    with _ctx(n, 2) as ctx:
        ref, st_ref = ctx.solve(psi, B, step=7)
    with _ctx(n, 2) as ctx:
        filler = _fill()
        S, st = ctx.solve(psi, B, step=7)
        del filler
        torch.cuda.empty_cache()
    assert st == st_ref and torch.equal(S, ref)
