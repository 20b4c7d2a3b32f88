"""Samples with a ragged nx and power-of-two ny, nz that step on the general x
passes because a carried x would cost more planes than it gains: one of each
line of the rule, with neighbours that are carried, against the oracle (1e-5 of
the fields, 1e-4 of what the steps change)."""
import numpy as np
import pytest

from oracle import demag as D
from oracle import llg as L
from paper_1406_7459_gb300 import inputs
from tests._helpers import oracle_spectrum, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MS, A_EX, CELL, HEXT, DT = 8.6e5, 1.3e-11, (4e-9, 3e-9, 5e-9), (1e4, -5e3, 2e3), 2e-14


@pytest.mark.parametrize("grid", [(147, 128, 8), (179, 128, 8), (643, 16, 32), (643, 16, 16), (768, 512, 2), (320, 128, 8),
                                  (387, 16, 64), (97, 512, 8), (106, 512, 8), (773, 16, 32), (193, 64, 32)])
def test_fields_and_steps_on_either_side_of_the_rule(grid):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1406_7459_gb300 import mm
    M = inputs.random_unit_m(grid, MS, seed=sum(grid))
    ctx = mm.mm_create(grid, CELL, MS, A_EX, 2e4, 0.2, inputs.GAMMA0)
    mm.mm_set_field(ctx, HEXT)
    Md = torch.from_numpy(M.reshape(-1)).cuda()
    out = torch.full_like(Md, float("nan"))
    Kt, Lp = oracle_spectrum(grid, CELL)
    M64 = M.astype(np.float64)

    def host(t):
        return t.cpu().numpy().reshape(M.shape).astype(np.float64)

    mm.mm_effective_field(ctx, Md, out)
    assert rel_l2(host(out), L.h_effective(M64, CELL, MS, A_EX, 2e4, HEXT, D.demag_fft(M64, Kt, Lp))) < 1e-5
    args = (CELL, MS, A_EX, 2e4, 0.2, inputs.GAMMA0, HEXT, Kt, Lp)
    mm.mm_set_m(ctx, Md)
    mm.mm_step(ctx, 2, DT)
    mm.mm_set_integrator(ctx, "heun")
    mm.mm_step(ctx, 1, DT)
    mm.mm_get_m(ctx, out)
    mm.mm_sync(ctx)
    ref = L.run_rk(L.run_euler(M64, 2, DT, *args), 1, DT, "heun", *args)
    assert rel_l2(host(out) - M64, ref - M64) < 1e-4
