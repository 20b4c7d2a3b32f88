"""Ragged samples: sides that are no powers of two, carried in the compile-time
transform lengths of the two-kernel step and of the split pass.  Sizes sit just above and at the
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


# thick samples and planes beyond shared memory: every z column length (first
# and last layer count of it), one odd line, rows and lines past a tile
THICK = [(17, 33, 9), (33, 18, 16), (20, 49, 17), (40, 17, 24), (65, 20, 25), (16, 30, 33), (18, 20, 48), (9, 34, 49),
         (12, 17, 64), (17, 12, 65), (8, 10, 96), (10, 9, 97), (7, 18, 128), (100, 65, 10), (257, 20, 12),
         (20, 1000, 3), (33, 700, 4), (18, 513, 7), (17, 641, 8), (5, 300, 15)]


@pytest.mark.parametrize("grid", GRIDS + THICK)
def test_ragged_film_fields_and_steps(grid):
    from paper_1406_7459_gb300 import mm
    nx, ny, nz = grid
    cell = (4e-9, 3e-9, 5e-9)
    Ku, alpha, dt, Hext = 2e4, 0.2, 2e-14, (1e4, -5e3, 2e3)
    M = inputs.random_unit_m(grid, MS, seed=sum(grid))
    ctx = mm.mm_create(grid, cell, MS, A_EX, Ku, alpha, GAMMA)
    assert mm.mm_plan_info(ctx)[1] == (4 if grid in THICK else 2)
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


# planes of the large-plane kernel: each of its line lengths at its first and
# last line count, the fewest planes that take it, and the power-of-two ones
BIG = [(129, 257, 5), (130, 320, 8), (129, 321, 3), (130, 384, 7), (129, 385, 4), (129, 511, 8), (131, 513, 3),
       (129, 640, 6), (129, 641, 5), (130, 768, 3), (129, 769, 3), (129, 1023, 4), (256, 512, 4), (256, 512, 8),
       (256, 1024, 4)]


@pytest.mark.parametrize("grid", BIG)
def test_large_planes_field_and_steps(grid):
    """Field, Euler steps and a Heun step of films whose planes one block takes
    a line per warp at a time: two kernels, and the oracle's values."""
    from paper_1406_7459_gb300 import mm
    cell, Hext, dt = (4e-9, 3e-9, 5e-9), (1e4, -5e3, 2e3), 2e-14
    M = inputs.random_unit_m(grid, MS, seed=sum(grid))
    ctx = mm.mm_create(grid, cell, MS, A_EX, 2e4, 0.2, GAMMA)
    assert mm.mm_plan_info(ctx)[1] == 2
    mm.mm_set_field(ctx, Hext)
    Md = torch.from_numpy(M.reshape(-1)).cuda()
    out = torch.full_like(Md, float("nan"))
    Kt, Lp = oracle_spectrum(grid, cell)
    M64 = M.astype(np.float64)
    mm.mm_demag_field(ctx, Md, out)
    Hd = D.demag_fft(M64, Kt, Lp)
    got = out.cpu().numpy().reshape(Hd.shape)
    assert rel_l2(got, Hd) < 1e-5 and rel_max(got, Hd) < 1e-5
    mm.mm_set_m(ctx, Md)
    mm.mm_step(ctx, 2, dt)
    mm.mm_set_integrator(ctx, "heun")
    mm.mm_step(ctx, 1, dt)
    mm.mm_get_m(ctx, out)
    mm.mm_sync(ctx)
    args = (cell, MS, A_EX, 2e4, 0.2, GAMMA, Hext, Kt, Lp)
    ref = L.run_rk(L.run_euler(M64, 2, dt, *args), 1, dt, "heun", *args)
    assert rel_l2(out.cpu().numpy().reshape(ref.shape) - M64, ref - M64) < 1e-4


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


@pytest.mark.parametrize("method", ["heun", "rk4"])
@pytest.mark.parametrize("grid", [(21, 37, 3), (257, 9, 2), (19, 22, 11)])
def test_ragged_runge_kutta_and_pass_timing(method, grid):
    """Fused stages on ragged films and blocks, in runs that end inside and
    after a captured graph, with a field evaluation in between; then one step
    advanced by the timing entry point."""
    from paper_1406_7459_gb300 import mm
    cell, Hext, dt = (4e-9, 3e-9, 5e-9), (1e4, -5e3, 2e3), 5e-14
    M = inputs.random_unit_m(grid, MS, seed=5)
    ctx = mm.mm_create(grid, cell, MS, A_EX, 1e4, 0.2, GAMMA)
    mm.mm_set_integrator(ctx, method)
    mm.mm_set_field(ctx, Hext)
    Md = torch.from_numpy(M.reshape(-1)).cuda()
    out = torch.empty_like(Md)
    mm.mm_set_m(ctx, Md)
    mm.mm_step(ctx, 17, dt)
    mm.mm_effective_field(ctx, Md, out)
    mm.mm_step(ctx, 2, dt)
    mm.mm_set_integrator(ctx, "euler")
    mm.mm_time_passes(ctx, 1, dt)
    mm.mm_step(ctx, 1, dt)
    mm.mm_get_m(ctx, out)
    mm.mm_sync(ctx)
    Kt, Lp = oracle_spectrum(grid, cell)
    args = (dt, method, cell, MS, A_EX, 1e4, 0.2, GAMMA, Hext, Kt, Lp)
    ref = L.run_rk(M.astype(np.float64), 19, *args)
    ref = L.run_rk(ref, 2, dt, "euler", *args[2:])
    got = out.cpu().numpy().reshape(ref.shape)
    assert rel_l2(got - M, ref - M) < 1e-4
