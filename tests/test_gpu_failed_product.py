"""A product that fails to launch leaves nothing behind: the next solve packs its own operand.

The failure is made on the host: the context's stream is in a capture that a synchronisation has
invalidated, so every launch on it returns an error until the capture ends."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1501_05427_gb300 import ulisse as u
from paper_1501_05427_gb300 import workloads as w

pytestmark = pytest.mark.gpu

RELAXED = 2   # cudaStreamCaptureModeRelaxed


def _cudart():
    with open("/proc/self/maps") as f:
        path = next(line.split()[-1] for line in f if "libcudart.so" in line)
    return ctypes.CDLL(path)


@pytest.mark.parametrize("precision", [u.PREC_FP32, u.PREC_MIXED])
def test_solve_after_a_failed_product(precision):
    u.load()
    rt = _cudart()
    prob = w.census_like(n=3_001, seed=9)
    stream = torch.cuda.Stream()
    X, y = torch.from_numpy(prob.X).cuda(), torch.from_numpy(prob.y).cuda()
    V = torch.randn(9, prob.n, device="cuda").t()
    U = torch.empty(9, prob.n, device="cuda").t()
    B = torch.from_numpy(np.random.default_rng(1).choice([-1.0, 1.0], (prob.n, 9)).astype(np.float32)).cuda()
    torch.cuda.synchronize()
    with u.Context(X, y, u.ulisse_config_default(precision=precision, seed=3), stream=stream) as ctx:
        ref, _ = ctx.solve(prob.psi_true, B, step=2)
        ctx.kmv(prob.psi_true, V, out=U)
        torch.cuda.synchronize()
        h = ctypes.c_void_p(stream.cuda_stream)
        assert rt.cudaStreamBeginCapture(h, RELAXED) == 0
        assert rt.cudaStreamSynchronize(h) != 0      # not permitted: invalidates the capture
        with pytest.raises(u.UlisseError):
            ctx.kmv(prob.psi_true, V, out=U)
        graph = ctypes.c_void_p()
        assert rt.cudaStreamEndCapture(h, ctypes.byref(graph)) != 0
        rt.cudaGetLastError()
        S, _ = ctx.solve(prob.psi_true, B, step=2)
    assert torch.equal(S, ref)
