"""The rounding of the exchange field where the field is formed with the stencil
of Eq. (4) on M: ragged samples, and power-of-two films of 512 rows and four
layers.  H_eff - H_demag of a slowly varying state is the exchange field up to
rounding.  M_x stays within a factor of two, so that its second differences are
exact in FP32; those of the small components round twice per axis, to 2^-24 of
M_y, M_z at most.  The sum H_d + H_ex rounds to 2^-24 of it and the stencil's
factors and sums to fewer than ten times 2^-24 of H_ex.  A stencil folded into the tensor spectrum would carry the transforms'
rounding of M itself, several times 1e-7 Ms."""
import numpy as np
import pytest

from oracle import llg as L
from paper_1406_7459_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MS, A_EX, GAMMA, CELL = 8.6e5, 1.3e-11, inputs.GAMMA0, (4e-9, 4e-9, 4e-9)


@pytest.mark.parametrize("grid", [(256, 512, 4), (512, 512, 4), (129, 385, 4), (40, 36, 3), (20, 18, 11)])
def test_exchange_is_the_stencil_of_neighbouring_differences(grid):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1406_7459_gb300 import mm
    nx, ny, nz = grid
    j, i = np.mgrid[0:ny, 0:nx]
    a = 0.1 * np.cos(2 * np.pi * i / 64) * np.cos(2 * np.pi * j / 50)
    m = np.stack([np.cos(a), np.sin(a), 0.05 * np.cos(2 * np.pi * i / 90)])
    m /= np.sqrt((m * m).sum(0))
    M = np.ascontiguousarray(np.repeat(m[:, None], nz, 1) * MS, np.float32)
    ctx = mm.mm_create(grid, CELL, MS, A_EX, 0.0, 0.1, GAMMA)
    Md = torch.from_numpy(M.reshape(-1)).cuda()
    hd, he = torch.empty_like(Md), torch.empty_like(Md)
    mm.mm_demag_field(ctx, Md, hd)
    mm.mm_effective_field(ctx, Md, he)
    mm.mm_sync(ctx)
    hd, he = (t.cpu().numpy().reshape(M.shape).astype(np.float64) for t in (hd, he))
    ex = L.h_exchange(M.astype(np.float64), CELL, MS, A_EX)
    w = 2 * A_EX / (4e-7 * np.pi * MS ** 2) / CELL[0] ** 2
    bound = 2.0 ** -24 * (np.abs(he).max() + 10 * np.abs(ex).max() + 6 * w * np.abs(M[1:]).max())
    print("largest error %.2e Ms, bound %.2e Ms" % (np.abs(he - hd - ex).max() / MS, bound / MS))
    assert np.abs(he - hd - ex).max() <= bound


@pytest.mark.parametrize("grid", [(40, 36, 3), (129, 385, 4), (33, 50, 1), (20, 18, 11)])
def test_ragged_exchange_is_added_in_one_rounding(grid):
    """H_eff = fl(H_d + pexch lap), lap by FP32 multiply-adds.  The multiply-adds
    are evaluated here in FP64 and rounded once more, which is the same but for
    ties of the second rounding (one in 2^29 and fewer); a separately
    rounded product would differ in a quarter of the cells."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1406_7459_gb300 import mm
    M = inputs.random_unit_m(grid, MS, seed=2)
    ctx = mm.mm_create(grid, CELL, MS, A_EX, 0.0, 0.1, GAMMA)
    Md = torch.from_numpy(M.reshape(-1)).cuda()
    hd, he = torch.empty_like(Md), torch.empty_like(Md)
    mm.mm_demag_field(ctx, Md, hd)
    mm.mm_effective_field(ctx, Md, he)
    mm.mm_sync(ctx)
    hd, he = (t.cpu().numpy().reshape(M.shape) for t in (hd, he))

    def fma(a, b, c):
        return (a.astype(np.float64) * np.float64(b) + c).astype(np.float32)

    w, d2 = np.float32(2 * A_EX / (4e-7 * np.pi * MS * MS)), np.float32(1 / CELL[0] ** 2)
    P = np.pad(M, ((0, 0), (1, 1), (1, 1), (1, 1)), mode="edge")
    lap = np.float32(0)
    for axis in (3, 2, 1) if grid[2] > 1 else (3, 2):
        lo, hi = [slice(1, -1)] * 3, [slice(1, -1)] * 3
        lo[axis - 1], hi[axis - 1] = slice(0, -2), slice(2, None)
        second = fma(M, -2.0, P[(slice(None), *hi)]) + P[(slice(None), *lo)]
        lap = fma(second, d2, lap)
    assert np.mean(fma(lap, w, hd) != he) < 1e-3
