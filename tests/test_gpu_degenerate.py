"""Samples of single rows, columns and layers and of a few cells, which the
ragged kernels carry in 16: fields against the oracle to 1e-5, Euler and Heun
steps to 1e-4 of what they change (FP32 transforms against FP64, as for the
other grids)."""
import numpy as np
import pytest

from oracle import demag as D
from oracle import llg as L
from paper_1406_7459_gb300 import inputs
from tests._helpers import oracle_spectrum, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MS, A_EX, CELL, HEXT, DT = 8.6e5, 1.3e-11, (4e-9, 3e-9, 5e-9), (1e4, -5e3, 2e3), 2e-14


@pytest.mark.parametrize("grid", [(1, 1, 1), (2, 1, 1), (1, 2, 1), (1, 1, 2), (9, 1, 1), (1, 9, 1), (600, 1, 1),
                                  (1, 64, 1), (1, 200, 2), (1, 33, 4), (1, 1, 20), (1, 1, 100), (2, 3, 1), (3, 2, 60),
                                  (1023, 1, 2), (1, 1023, 3)])
def test_single_rows_columns_and_layers(grid):
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

    mm.mm_demag_field(ctx, Md, out)
    Hd = D.demag_fft(M64, Kt, Lp)
    assert rel_l2(host(out), Hd) < 1e-5
    mm.mm_effective_field(ctx, Md, out)
    assert rel_l2(host(out), L.h_effective(M64, CELL, MS, A_EX, 2e4, HEXT, Hd)) < 1e-5
    args = (CELL, MS, A_EX, 2e4, 0.2, inputs.GAMMA0, HEXT, Kt, Lp)
    mm.mm_set_m(ctx, Md)
    mm.mm_step(ctx, 4, DT)
    mm.mm_set_integrator(ctx, "heun")
    mm.mm_step(ctx, 2, DT)
    mm.mm_get_m(ctx, out)
    mm.mm_sync(ctx)
    ref = L.run_rk(L.run_euler(M64, 4, DT, *args), 2, DT, "heun", *args)
    assert rel_l2(host(out) - M64, ref - M64) < 1e-4
    E = mm.mm_energy(ctx)
    want = L.energy_terms(host(out), D.demag_fft(host(out), Kt, Lp), CELL, MS, A_EX, 2e4, HEXT)
    assert np.abs(E - want).max() <= 1e-5 * np.abs(want).max()
