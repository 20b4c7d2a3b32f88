"""Ragged films: sides that are no powers of two, carried in the compile-time
transform lengths of the two-kernel step.  Sizes sit just above and at the
carrier lengths (one row or cell into the next length, tiles with one valid
row, a full carrier), for every layer count and carrier length of the plane
and x kernels.  Tolerances are those of the other field and step tests: 1e-5
of the field, 1e-4 of what the steps change (FP32 transforms against FP64)."""
import numpy as np
import pytest

from oracle import demag as D
from oracle import llg as L
from paper_1406_7459_gb300 import inputs
from tests._helpers import oracle_spectrum, rel_l2, rel_max

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MS, A_EX, GAMMA = 8.6e5, 1.3e-11, inputs.GAMMA0


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


GRIDS = [(17, 33, 1), (33, 17, 2), (48, 50, 3), (49, 65, 4), (65, 97, 5), (97, 49, 6), (129, 30, 7), (193, 20, 8),
         (256, 18, 2), (257, 31, 4), (321, 257, 1), (385, 20, 3), (513, 21, 2), (641, 30, 1), (769, 33, 1),
         (1023, 19, 2), (20, 1023, 2), (19, 513, 3), (18, 641, 3), (30, 769, 1), (36, 321, 4), (40, 193, 5),
         (5, 129, 8), (9, 6, 1)]


@pytest.mark.parametrize("grid", GRIDS)
def test_ragged_film_fields_and_steps(grid):
    from paper_1406_7459_gb300 import mm
    nx, ny, nz = grid
    cell = (4e-9, 3e-9, 5e-9)
    Ku, alpha, dt, Hext = 2e4, 0.2, 2e-14, (1e4, -5e3, 2e3)
    M = inputs.random_unit_m(grid, MS, seed=sum(grid))
    ctx = mm.mm_create(grid, cell, MS, A_EX, Ku, alpha, GAMMA)
    assert mm.mm_plan_info(ctx)[1] == 2
    mm.mm_set_field(ctx, Hext)
    Md = torch.from_numpy(M.reshape(-1)).cuda()
    out = torch.full_like(Md, float("nan"))
    Kt, Lp = oracle_spectrum(grid, cell)
    M64 = M.astype(np.float64)

    def host(t):
        return t.cpu().numpy().reshape(3, nz, ny, nx).astype(np.float64)

    mm.mm_demag_field(ctx, Md, out)
    Hd = D.demag_fft(M64, Kt, Lp)
    assert rel_l2(host(out), Hd) < 1e-5 and rel_max(host(out), Hd) < 1e-5
    mm.mm_effective_field(ctx, Md, out)
    assert rel_l2(host(out), L.h_effective(M64, cell, MS, A_EX, Ku, Hext, Hd)) < 1e-5
    mm.mm_set_m(ctx, Md)
    mm.mm_step(ctx, 18, dt)                       # a 16-step graph, then single launches
    mm.mm_get_m(ctx, out)
    mm.mm_sync(ctx)
    ref = L.run_euler(M64, 18, dt, cell, MS, A_EX, Ku, alpha, GAMMA, Hext, Kt, Lp)
    assert rel_l2(host(out) - M64, ref - M64) < 1e-4


def test_ragged_spectrum_is_formed_on_demand():
    """The stored-spectrum entry points of a ragged film, whose steps do not
    read that spectrum: the same padded lengths and values as the oracle's,
    before and after steps, and usable for the allocation-free field."""
    from paper_1406_7459_gb300 import mm
    grid, cell = (21, 13, 3), (4e-9, 3e-9, 5e-9)
    ctx = mm.mm_create(grid, cell, MS, A_EX, 0.0, 0.5, GAMMA)
    (Lx, Ly, Lz), _ = mm.mm_plan_info(ctx)
    M = torch.from_numpy(inputs.random_unit_m(grid, MS, 3).reshape(-1)).cuda()
    mm.mm_set_m(ctx, M)
    mm.mm_step(ctx, 2, 1e-14)
    Kt = torch.empty((Lx // 2 + 1) * (Lz // 2 + 1) * (Ly // 2 + 1) * 6, device="cuda")
    mm.mm_kernel_spectrum(ctx, Kt)
    a, b = torch.empty_like(M), torch.empty_like(M)
    mm.mm_demag_field(ctx, M, a)
    mm.mm_demag_field_noalloc(grid, Kt, M, b)
    torch.cuda.synchronize()
    assert rel_l2(a.cpu().numpy().astype(np.float64), b.cpu().numpy().astype(np.float64)) < 1e-5
