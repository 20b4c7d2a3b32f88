"""Tiled x-step copies on a film whose planes the large-plane kernel takes: the
tensor maps concern the x-step kernel alone, so they are there wherever its box
fits, and every mask gives the default copies' bits."""
import numpy as np
import pytest

from paper_1406_7459_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_tiled_copies_on_large_planes_are_bitwise_the_default():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1406_7459_gb300 import mm
    grid = (256, 512, 4)
    M = torch.from_numpy(np.ascontiguousarray(inputs.perturbed_m(grid, 8.6e5, seed=4, amplitude=0.3),
                                              np.float32).reshape(-1)).cuda()
    got = []
    for mask in (0, mm.MM_TILED_GATHER, mm.MM_TILED_SCATTER, mm.MM_TILED_GATHER | mm.MM_TILED_SCATTER):
        ctx = mm.mm_create(grid, (4e-9,) * 3, 8.6e5, 1.3e-11, 5e2, 0.02, inputs.GAMMA0)
        mm.mm_set_tiled_copies(ctx, mask)
        assert mm.mm_get_tiled_copies(ctx) == mask
        mm.mm_set_m(ctx, M)
        mm.mm_step(ctx, 3, 5e-14)
        out = torch.empty_like(M)
        mm.mm_get_m(ctx, out)
        mm.mm_sync(ctx)
        got.append(out.cpu().numpy())
    assert np.all(np.isfinite(got[0]))
    assert all(np.array_equal(g, got[0]) for g in got[1:])


def test_tiled_copies_stay_refused_where_planes_are_split():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1406_7459_gb300 import mm
    for grid in ((256, 512, 8), (64, 64, 32), (512, 512, 4)):
        ctx = mm.mm_create(grid, (4e-9,) * 3, 8.6e5, 1.3e-11, 5e2, 0.02, inputs.GAMMA0)
        with pytest.raises(mm.MMError) as e:
            mm.mm_set_tiled_copies(ctx, mm.MM_TILED_GATHER)
        assert e.value.code == mm.MM_EUNSUPPORTED
