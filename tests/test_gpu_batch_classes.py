"""The batch's size classes: samples at the edges of every class of the
ragged-film kernels and samples of the general kernels in one batch, against
the FP64 oracle (1e-5 of the state, as for the other batch tests) and, bit
for bit, between the graph and the persistent step; and batches of different
shapes alive at once."""
import numpy as np
import pytest

from oracle import llg as L
from paper_1406_7459_gb300 import inputs
from tests._helpers import oracle_spectrum, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MS, A_EX, CELL, DT = 8.6e5, 1.3e-11, (5e-9, 4e-9, 3e-9), 5e-14
# last row / cell of one class, first of the next; four layers; then general
# kernels: a long row, three layers of long lines, a side above every class
CLASSES = [(16, 16, 1), (17, 16, 2), (32, 17, 3), (33, 32, 4), (48, 33, 1), (49, 48, 2), (64, 49, 3), (65, 64, 4),
           (96, 65, 1), (97, 96, 2), (128, 97, 2), (129, 128, 1), (192, 129, 1), (193, 192, 2), (256, 193, 1),
           (255, 256, 2), (3, 5, 2), (1, 9, 1)]
GENERAL = [(257, 12, 1), (20, 65, 3), (12, 257, 1)]


def _batch(grids):
    from paper_1406_7459_gb300 import mm
    n = len(grids)
    b = mm.mm_batch_create(grids, [CELL] * n, [MS] * n, [A_EX] * n, [1e4] * n, [0.2] * n, [inputs.GAMMA0] * n)
    mm.mm_batch_set_field(b, [(2e4, -1e4, 5e3)] * n)
    M = [inputs.random_unit_m(g, MS, 10 + i) for i, g in enumerate(grids)]
    mm.mm_batch_set_m(b, torch.from_numpy(np.concatenate([v.reshape(-1) for v in M])).cuda())
    return b, M


def _state(b):
    from paper_1406_7459_gb300 import mm
    out = torch.empty(b.total, device="cuda")
    mm.mm_batch_get_m(b, out)
    mm.mm_batch_sync(b)
    return out.cpu().numpy()


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("grids", [CLASSES, GENERAL, CLASSES[::3] + GENERAL], ids=["classes", "general", "mixed"])
def test_batch_classes_match_oracle_on_both_paths(grids):
    from paper_1406_7459_gb300 import mm
    b, M = _batch(grids)
    mm.mm_batch_step(b, 3, DT)
    got = _state(b)
    p, _ = _batch(grids)
    mm.mm_batch_set_path(p, mm.MM_STEP_PERSISTENT)
    mm.mm_batch_step(p, 3, DT)
    assert np.array_equal(_state(p), got)
    for i, g in enumerate(grids):
        Kt, Lp = oracle_spectrum(g, CELL)
        ref = L.run_euler(M[i].astype(np.float64), 3, DT, CELL, MS, A_EX, 1e4, 0.2, inputs.GAMMA0,
                          (2e4, -1e4, 5e3), Kt, Lp)
        mine = got[b.offsets[i]:b.offsets[i + 1]].reshape(ref.shape)
        assert rel_l2(mine, ref) < 1e-5, g


def test_batches_of_different_shapes_alive_together():
    """A later batch with smaller tiles does not take the first one's shared
    memory away, on the class kernels or (long rows) the general ones."""
    from paper_1406_7459_gb300 import mm
    big, _ = _batch([(256, 256, 2), (700, 40, 2)])
    mm.mm_batch_autotune(big, DT)
    small, _ = _batch([(20, 20, 1), (300, 8, 1)])
    mm.mm_batch_autotune(small, DT)
    mm.mm_batch_step(big, 2, DT)
    mm.mm_batch_step(small, 2, DT)
    assert np.all(np.isfinite(_state(big))) and np.all(np.isfinite(_state(small)))
