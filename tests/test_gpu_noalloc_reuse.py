"""dir_register_noalloc after a call of another size: its static scratch holds
whatever that call left, which no result may depend on."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", [{}, {"plain_kernels": 1}, {"fuse": 3}, {"fuse": 1},
                                  {"precision": 4}], ids=str)
@pytest.mark.parametrize("dims,levels", [((1, 40, 6), 1), ((2, 5, 4), 2), ((3, 30, 9), 3),
                                         ((1, 1, 1), 1), ((64, 1, 3), 2)], ids=str)
def test_narrow_volume_after_a_call_that_left_nan(dims, levels, form):
    """On an x axis of one voxel the gathers read row padding with weight 0."""
    import paper_0909_0928_gb300 as dl

    big = torch.full((32, 64, 64), float("nan"), device="cuda")
    left = torch.empty((3, 32, 64, 64), device="cuda")
    g = torch.Generator(device="cuda").manual_seed(3)
    S, M = (100.0 * torch.rand(dims[::-1], generator=g, device="cuda") for _ in range(2))
    out = torch.empty((3,) + dims[::-1], device="cuda")
    for variant in (0, 2, 5):
        dl.dir_register_noalloc(big, big, (64, 64, 32), variant,
                                dl.dir_params_default(levels=1, iters=[2]), left)
        p = dl.dir_params_default(levels=levels, iters=[3] * levels, **form)
        dl.dir_register_noalloc(S, M, dims, variant, p, out)
        ctx = dl.dir_create(S, M, dims, (1.0, 1.0, 1.0), dl.DIR_F32, True, variant, p)
        dl.dir_register(ctx)
        want = dl.dir_get_field(ctx, np.empty(out.shape, np.float32))
        dl.dir_destroy(ctx)
        assert np.isfinite(want).all()
        assert np.array_equal(out.cpu().numpy(), want), variant
