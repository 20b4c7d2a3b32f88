"""Sequences of calls on one context or batch, where one call leaves state that
the next one uses: the integrators one after the other, a field changed with
steps in flight, long persistent launches.  Tolerances are those of the step
tests: 1e-4 of what the steps change against the FP64 oracle, bit equality
between two forms of the same arithmetic."""
import numpy as np
import pytest

from oracle import llg as L
from paper_1406_7459_gb300 import inputs
from tests._helpers import oracle_spectrum, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MS, A_EX, GAMMA = 8.6e5, 1.3e-11, inputs.GAMMA0
CELL, HEXT = (4e-9, 3e-9, 5e-9), (1e4, -5e3, 2e3)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("method", ["heun", "rk4"])
@pytest.mark.parametrize("grid", [(20, 12, 3), (32, 32, 2), (700, 540, 1), (1100, 6, 1)])
def test_runge_kutta_after_an_adaptive_run(method, grid):
    """An adaptive run allocates the stage state alone; Heun and RK4 also need
    the sum of their slopes.  Fused stages (ragged and power-of-two), a film
    above the fused stages' size and the general kernels."""
    from paper_1406_7459_gb300 import mm
    M = np.ascontiguousarray(inputs.perturbed_m(grid, MS, seed=3, amplitude=0.3), np.float32)
    ctx = mm.mm_create(grid, CELL, MS, A_EX, 1e4, 0.2, GAMMA)
    mm.mm_set_field(ctx, HEXT)
    Md = torch.from_numpy(M.reshape(-1)).cuda()
    mm.mm_set_m(ctx, Md)
    done, _, _ = mm.mm_run_adaptive(ctx, 1e-14, 1e-14, 1.0, 4)
    assert done
    mid = torch.empty_like(Md)
    mm.mm_get_m(ctx, mid)
    mm.mm_set_integrator(ctx, method)
    mm.mm_step(ctx, 2, 2e-14)
    out = torch.empty_like(Md)
    mm.mm_get_m(ctx, out)
    mm.mm_sync(ctx)
    Kt, Lp = oracle_spectrum(grid, CELL)
    m64 = mid.cpu().numpy().reshape(M.shape).astype(np.float64)
    ref = L.run_rk(m64, 2, 2e-14, method, CELL, MS, A_EX, 1e4, 0.2, GAMMA, HEXT, Kt, Lp)
    assert rel_l2(out.cpu().numpy().reshape(M.shape) - m64, ref - m64) < 1e-4


def _batch(grids, stream=None):
    from paper_1406_7459_gb300 import mm
    n = len(grids)
    b = mm.mm_batch_create(grids, [CELL] * n, [MS] * n, [A_EX] * n, [1e4] * n, [0.2] * n, [GAMMA] * n, stream=stream)
    mm.mm_batch_set_field(b, [HEXT] * n)
    M = np.concatenate([inputs.random_unit_m(g, MS, 20 + i).reshape(-1) for i, g in enumerate(grids)])
    Md = torch.from_numpy(M).cuda()
    torch.cuda.synchronize()
    mm.mm_batch_set_m(b, Md)
    return b


def _batch_state(b):
    from paper_1406_7459_gb300 import mm
    out = torch.empty(b.total, device="cuda")
    mm.mm_batch_get_m(b, out)
    mm.mm_batch_sync(b)
    return out.cpu().numpy()


@pytest.mark.parametrize("grids", [[(33, 17, 2), (16, 48, 1), (100, 30, 2), (200, 64, 1), (64, 64, 4)],
                                   [(257, 12, 1), (20, 65, 3)], [(40, 40, 1), (12, 257, 1)]],
                         ids=["classes", "general", "mixed"])
def test_long_persistent_launch_is_bitwise_the_batched_kernels(grids):
    """One launch of 48 steps rewrites each state buffer 24 times between its
    barriers; the batched kernels read a buffer that no running kernel
    writes."""
    from paper_1406_7459_gb300 import mm
    got = []
    for path in (mm.MM_STEP_GRAPH, mm.MM_STEP_PERSISTENT):
        b = _batch(grids)
        mm.mm_batch_set_path(b, path)
        mm.mm_batch_step(b, 48, 5e-14)
        got.append(_batch_state(b))
    assert np.all(np.isfinite(got[0]))
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("path", ["graph", "persistent"])
@pytest.mark.parametrize("general", [False, True])
def test_batch_field_change_behind_steps_in_flight(path, general):
    """mm_batch_step returns with its kernels in flight; on a stream that the
    legacy stream does not wait for, a field set right after it must reach
    the later steps only."""
    from paper_1406_7459_gb300 import mm
    grids = [(400, 40, 2)] * 24 if general else [(256, 64, 2)] * 60
    got = []
    for wait in (True, False):
        side = torch.cuda.Stream()
        b = _batch(grids, side)
        if path == "persistent":
            mm.mm_batch_set_path(b, mm.MM_STEP_PERSISTENT)
        for n, k in ((60, -1.0), (20, 0.5)):
            mm.mm_batch_step(b, n, 5e-14)
            if wait:
                side.synchronize()
            mm.mm_batch_set_field(b, [tuple(k * h for h in HEXT)] * len(grids))
        mm.mm_batch_step(b, 3, 5e-14)
        got.append(_batch_state(b))
    assert np.all(np.isfinite(got[0]))
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("first,second", [((1100, 40, 4), (1030, 3, 4)), ((1100, 24, 12), (1040, 3, 9))])
def test_general_contexts_of_different_sizes_alive_together(first, second):
    """The general kernels' shared memory follows the sample; a context created
    later with shorter lines leaves an earlier one its own."""
    from paper_1406_7459_gb300 import mm

    def make(grid):
        ctx = mm.mm_create(grid, CELL, MS, A_EX, 1e4, 0.2, GAMMA)
        mm.mm_set_m(ctx, torch.from_numpy(inputs.random_unit_m(grid, MS, 5).reshape(-1)).cuda())
        return ctx

    got = []
    for shared in (False, True):
        ctx = make(first)
        other = make(second) if shared else None
        if shared:
            mm.mm_step(other, 1, 2e-14)
        mm.mm_step(ctx, 2, 2e-14)
        out = torch.empty(3 * ctx.N, device="cuda")
        mm.mm_get_m(ctx, out)
        mm.mm_sync(ctx)
        got.append(out)
    assert torch.isfinite(got[0]).all() and torch.equal(got[0], got[1])
