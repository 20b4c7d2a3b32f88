"""The scale of H_demag on carrier lengths.  Random rounding averages out of the
projection <H, H_exact> / <H_exact, H_exact>; what would stay is a common
factor, the transforms' gains with their rounded constants, by which the
spectrum is divided.  The gains spread by 2.4e-8 and less over the wavenumbers of
an axis, which bounds what a wrong weighting of them could leave of a random
state.  Without the division these grids lose 1.2e-7 to 1.8e-7."""
import numpy as np
import pytest

from oracle import demag as D
from paper_1406_7459_gb300 import inputs
from tests._helpers import oracle_spectrum

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MS, CELL = 8.6e5, (4e-9, 4e-9, 4e-9)


@pytest.mark.parametrize("grid", [(100, 80, 20), (90, 90, 12), (40, 700, 1), (500, 90, 2), (90, 40, 90)])
def test_demag_field_of_ragged_samples_keeps_its_scale(grid):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1406_7459_gb300 import mm
    M = inputs.random_unit_m(grid, MS, seed=6)
    ctx = mm.mm_create(grid, CELL, MS, 1.3e-11, 0.0, 0.1, inputs.GAMMA0)
    Md = torch.from_numpy(M.reshape(-1)).cuda()
    out = torch.empty_like(Md)
    mm.mm_demag_field(ctx, Md, out)
    mm.mm_sync(ctx)
    Kt, Lp = oracle_spectrum(grid, CELL)
    ref = D.demag_fft(M.astype(np.float64), Kt, Lp)
    got = out.cpu().numpy().reshape(ref.shape).astype(np.float64)
    scale = float((got * ref).sum() / (ref * ref).sum()) - 1.0
    print("%s: scale error %.2e" % (grid, scale))
    assert abs(scale) < 2.4e-8 * (3 if grid[2] > 8 else 2)


@pytest.mark.parametrize("grid", [(150, 361, 8), (300, 90, 2), (90, 90, 12), (700, 65, 1), (30, 40, 20)])
def test_scale_of_smooth_states(grid):
    """A state near saturation, whose field comes from the smallest wavenumbers:
    their transforms hold few of the rounded constants, 0 and 1 none, so a common
    factor for all wavenumbers would put this field off by up to 1.4e-7.  What
    remains is the rounding of the few tensor entries it rests on, 2^-25
    each, and of M."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1406_7459_gb300 import mm
    M = np.ascontiguousarray(inputs.perturbed_m(grid, MS, seed=6, amplitude=0.02), np.float32)
    ctx = mm.mm_create(grid, CELL, MS, 1.3e-11, 0.0, 0.1, inputs.GAMMA0)
    Md = torch.from_numpy(M.reshape(-1)).cuda()
    out = torch.empty_like(Md)
    mm.mm_demag_field(ctx, Md, out)
    mm.mm_sync(ctx)
    Kt, Lp = oracle_spectrum(grid, CELL)
    ref = D.demag_fft(M.astype(np.float64), Kt, Lp)
    got = out.cpu().numpy().reshape(ref.shape).astype(np.float64)
    scale = float((got * ref).sum() / (ref * ref).sum()) - 1.0
    print("%s: scale error %.2e" % (grid, scale))
    assert abs(scale) < 2.0 ** -24
