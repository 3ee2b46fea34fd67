"""dir_autotune chooses among the launches that the levels run."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _tuned(dims, variant, levels, reps=3):
    import paper_0909_0928_gb300 as dl

    g = torch.Generator(device="cuda").manual_seed(5)
    S, M = (100.0 * torch.rand(dims[::-1], generator=g, device="cuda") for _ in range(2))
    p = dl.dir_params_default(levels=levels, iters=[4] * levels)
    ctx = dl.dir_create(S, M, dims, (1.0, 1.0, 1.0), dl.DIR_F32, True, variant, p)
    try:
        dl.dir_register(ctx)
        before = dl.dir_get_field(ctx, np.empty((3,) + dims[::-1], np.float32))
        shapes = dl.dir_autotune(ctx, reps, levels)
        dl.dir_register(ctx)
        after = dl.dir_get_field(ctx, np.empty((3,) + dims[::-1], np.float32))
        assert np.array_equal(after, before)
        return shapes
    finally:
        dl.dir_destroy(ctx)


@pytest.mark.parametrize("variant", [0, 2, 5])
def test_resident_levels_have_no_shape(variant):
    assert _tuned((32, 32, 16), variant, 3) == [(2, 0)] * 3


@pytest.mark.parametrize("variant", [3, 5])
def test_depths_without_u_in_the_scratch(variant):
    """128 x 120 x 90 is above 2^20 voxels: two depths, and strips in y, of which
    18 boxes of seven rows are as long as 120 rows and six of halo."""
    for _ in range(3):
        depth, boxes = _tuned((128, 120, 90), variant, 1)[0]
        assert depth in (4, 8)
        assert boxes == 0 or 2 <= boxes <= 18
