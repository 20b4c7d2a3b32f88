"""Captured graphs against launches one by one, on runs that are long enough to
capture: a context launches its first 128 steps of a dt directly, a batch its
first 8.  Replayed steps must have the direct launches' bits on every kind of
plan and integrator, after the field or the copies changed and between two
runs; the launch form says that a graph was in fact replayed."""
import numpy as np
import pytest

from paper_1406_7459_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MS, A_EX, GAMMA, CELL = 8.6e5, 1.3e-11, inputs.GAMMA0, (4e-9, 3e-9, 5e-9)
WARM = 128


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


# ragged film, ragged block, power-of-two film and block, planes of the
# large-plane kernel (both kinds), general kernels (whose single Runge-Kutta
# steps are graphs too); Runge-Kutta stages fused and unfused
RUNS = [((20, 12, 3), "euler"), ((19, 22, 11), "euler"), ((32, 32, 2), "euler"), ((32, 32, 32), "euler"),
        ((256, 512, 4), "euler"), ((129, 385, 4), "euler"), ((1100, 6, 1), "euler"), ((20, 12, 3), "rk4"),
        ((32, 32, 2), "heun"), ((19, 22, 11), "rk4"), ((700, 540, 1), "rk4"), ((1100, 6, 1), "heun")]


@pytest.mark.parametrize("grid,method", RUNS)
def test_replayed_steps_are_bitwise_direct_launches(monkeypatch, grid, method):
    from paper_1406_7459_gb300 import mm
    M = torch.from_numpy(np.ascontiguousarray(inputs.perturbed_m(grid, MS, seed=9, amplitude=0.3), np.float32)
                         .reshape(-1)).cuda()
    got = []
    for direct in ("0", "1"):
        monkeypatch.setenv("MM_NO_GRAPHS", direct)
        ctx = mm.mm_create(grid, CELL, MS, A_EX, 1e4, 0.1, GAMMA)
        mm.mm_set_integrator(ctx, method)
        mm.mm_set_m(ctx, M)
        states, forms = [], []
        for n in (WARM + 37, 16, 21):             # graphs from both parities, then both kinds again
            mm.mm_step(ctx, n, 2e-14)
            forms.append(mm.mm_step_form(ctx))
        states.append(mm.mm_get_m(ctx, torch.empty_like(M)))
        mm.mm_set_field(ctx, (2e3, -1e3, 5e2))    # captured anew with the new field
        mm.mm_step(ctx, WARM + 16, 2e-14)
        forms.append(mm.mm_step_form(ctx))
        states.append(mm.mm_get_m(ctx, torch.empty_like(M)))
        mm.mm_sync(ctx)
        got.append([s.cpu().numpy() for s in states])
        if direct == "1":
            assert forms == [mm.MM_FORM_DIRECT] * 4
        else:
            assert all(f & mm.MM_FORM_GRAPH for f in forms)
    assert np.all(np.isfinite(got[0][1]))
    assert not np.array_equal(got[0][0], got[0][1])
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])


def test_tiled_copies_switched_between_replays():
    from paper_1406_7459_gb300 import mm
    grid = (64, 64, 4)
    M = torch.from_numpy(np.ascontiguousarray(inputs.perturbed_m(grid, MS, seed=4, amplitude=0.3), np.float32)
                         .reshape(-1)).cuda()
    got = []
    for mask in (0, mm.MM_TILED_GATHER | mm.MM_TILED_SCATTER):
        ctx = mm.mm_create(grid, CELL, MS, A_EX, 1e4, 0.1, GAMMA)
        mm.mm_set_m(ctx, M)
        mm.mm_step(ctx, WARM + 16, 2e-14)
        assert mm.mm_step_form(ctx) & mm.MM_FORM_GRAPH
        mm.mm_set_tiled_copies(ctx, mask)
        mm.mm_step(ctx, WARM + 32, 2e-14)
        assert mm.mm_step_form(ctx) & mm.MM_FORM_GRAPH
        got.append(mm.mm_get_m(ctx, torch.empty_like(M)))
        mm.mm_sync(ctx)
    assert torch.equal(got[0], got[1])


def test_batch_replay_is_bitwise_direct_launches():
    """Every class of kernels side by side and the general ones; a field set
    before each step keeps the reference on direct launches."""
    from paper_1406_7459_gb300 import mm
    grids = [(nx, ny, nz) for nx, ny in ((16, 16), (30, 32), (48, 40), (60, 64)) for nz in (1, 2, 3, 4)]
    grids += [(90, 90, 1), (120, 128, 2), (190, 180, 2), (250, 256, 1), (300, 12, 1), (20, 65, 3)]
    n, field = len(grids), [(1e4, -5e3, 2e3)] * len(grids)
    M = torch.from_numpy(np.concatenate([inputs.random_unit_m(g, MS, 30 + i).reshape(-1)
                                         for i, g in enumerate(grids)])).cuda()
    got = []
    for direct in (False, True):
        b = mm.mm_batch_create(grids, [CELL] * n, [MS] * n, [A_EX] * n, [1e4] * n, [0.2] * n, [GAMMA] * n)
        mm.mm_batch_set_field(b, field)
        mm.mm_batch_set_m(b, M)
        for k in (11, 6):
            for _ in range(k if direct else 1):
                if direct:
                    mm.mm_batch_set_field(b, field)
                mm.mm_batch_step(b, 1 if direct else k, 2e-14)
            assert mm.mm_batch_launch_form(b) == (3 if direct else 0)
        got.append(mm.mm_batch_get_m(b, torch.empty_like(M)))
        mm.mm_batch_sync(b)
    assert torch.isfinite(got[0]).all()
    assert torch.equal(got[0], got[1])
