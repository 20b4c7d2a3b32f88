"""The renormalisation to |M| = Ms.  With a time step below the rounding of every
cell the new state is M Ms / |M|, which can be followed rounding by rounding:
|M|^2 by multiply-adds from z to x, so that the largest square (the easy axis
is x) enters unrounded."""
import numpy as np
import pytest

from paper_1406_7459_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MS = np.float32(8.6e5)


@pytest.mark.parametrize("method", ["euler", "heun", "rk4"])
@pytest.mark.parametrize("grid", [(40, 36, 3), (33, 50, 1), (20, 18, 11)])
def test_ragged_renormalisation_rounds_the_sum_once(grid, method):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1406_7459_gb300 import mm
    M = (inputs.perturbed_m(grid, MS, seed=8, amplitude=0.1) * 1.00001).astype(np.float32)
    ctx = mm.mm_create(grid, (4e-9,) * 3, float(MS), 1.3e-11, 0.0, 0.1, inputs.GAMMA0)
    mm.mm_set_integrator(ctx, method)
    Md = torch.from_numpy(np.ascontiguousarray(M).reshape(-1)).cuda()
    mm.mm_set_m(ctx, Md)
    mm.mm_step(ctx, 1, 1e-30)
    out = torch.empty_like(Md)
    mm.mm_get_m(ctx, out)
    mm.mm_sync(ctx)

    def fma(a, b, c):                     # a second rounding ties once in 2^29
        return (a.astype(np.float64) * b + c).astype(np.float32)

    n2 = fma(M[0], M[0], fma(M[1], M[1], M[2] * M[2]))
    want = M * (MS / np.sqrt(n2))
    assert want.dtype == np.float32
    assert np.mean(out.cpu().numpy().reshape(M.shape) != want) < 1e-3
