"""FP32 launch tables (ulisse_set_tune): an entry with rows per thread is the SIMT kernel in that shape,
with or without a forced split; one without is the untuned choice.  Products in the same form are
equal bit for bit; the autotuner's own table gives the tuned context's products when installed."""
import numpy as np
import pytest
import torch

from paper_1501_05427_gb300 import ulisse as u
from paper_1501_05427_gb300 import workloads as w

pytestmark = pytest.mark.gpu


def _ctx(prob, **cfg):
    return u.Context(torch.from_numpy(prob.X).cuda(), torch.from_numpy(prob.y).cuda(),
                     u.ulisse_config_default(**cfg))


def _entry(width, rows, nsplit=0):
    return {"width": width, "rows_per_thread": rows, "nsplit": nsplit, "cross_term": 0}


@pytest.mark.parametrize("rows", [2, 4])
def test_entry_fixes_the_simt_shape(rows):
    prob = w.census_like(n=3_001, seed=31)
    V = torch.randn(17, prob.n, device="cuda", generator=torch.Generator("cuda").manual_seed(1)).t()
    with _ctx(prob, kmv_rows_per_thread=rows) as ctx:
        simt = ctx.kmv(prob.psi_true, V).clone()
    with _ctx(prob) as ctx:
        untuned = ctx.kmv(prob.psi_true, V).clone()
        assert not torch.equal(untuned, simt)    # the sizes where the tensor cores take it
        ctx.set_tune([_entry(k + 1, rows) for k in range(17)])
        assert torch.equal(ctx.kmv(prob.psi_true, V), simt)
        ctx.set_tune([_entry(k + 1, 0) for k in range(17)])
        assert torch.equal(ctx.kmv(prob.psi_true, V), untuned)
        for bad in (_entry(1, 0, nsplit=2), _entry(1, 3), _entry(0, 0)):
            with pytest.raises(u.UlisseError):
                ctx.set_tune([bad])


def test_installed_table_reproduces_the_tuned_context():
    prob = w.census_like(n=12_000, seed=32)
    Vs = [torch.randn(R, prob.n, device="cuda").t() for R in (1, 5, 9, 17)]
    with _ctx(prob) as ctx:
        table = ctx.autotune(prob.psi_true, 17, reps=2)
        outs = [ctx.kmv(prob.psi_true, V).clone() for V in Vs]
    with _ctx(prob) as ctx:
        ctx.set_tune(table)
        for V, ref in zip(Vs, outs):
            assert torch.equal(ctx.kmv(prob.psi_true, V), ref)


def test_tuned_splits_can_be_installed():
    # 50,000 points, one column: the plan's split is 49, its double beyond the 64 of a table
    prob = w.census_like(n=50_000, seed=33)
    with _ctx(prob) as ctx:
        table = ctx.autotune(prob.psi_true, 2, reps=1)
        ctx.set_tune(table)
        ctx.set_tune([dict(e, rows_per_thread=2, nsplit=64) for e in table])
    assert all(0 <= e["nsplit"] <= 64 for e in table)
