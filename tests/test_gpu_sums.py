"""The sums of an iteration (dir_get_history) and the stop test that reads them,
where rounding or the ends of the float range show: what the plain-load kernels
report, whichever kernels a level runs.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

# default: a resident level; fuse 4: the split kernels
FORMS = {"resident": {}, "split": {"fuse": 4}}


@pytest.fixture(scope="module")
def dl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0909_0928_gb300 as dl
    return dl


def _register(dl, S, M, variant, n, start=None, **kw):
    u0 = None if start is None else torch.tensor(np.ascontiguousarray(start)).cuda()
    p = dl.dir_params_default(levels=1, iters=[n], alpha=0.7, init_field=u0, **kw)
    ctx = dl.dir_create(S, M, S.shape[::-1], (1.0, 1.0, 1.0), dl.DIR_F32, False, variant, p)
    try:
        st = dl.dir_register(ctx)
        return st.iters_run[0], dl.dir_get_history(ctx, n)
    finally:
        dl.dir_destroy(ctx)


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("value", [1e25, 1e19, 3.7, 0.1, 1e-3, 1e-18, 1e-20, 1e-21, 1e-24, 0.0,
                                   np.inf, np.nan], ids=str)
def test_norms_of_one_voxel(dl, value, form):
    """A sum over one voxel is that voxel's norm, so it has to be the plain
    kernels' bit for bit: squares that overflow (not a number, so that no stop
    test takes them for convergence), that are subnormal, that underflow."""
    S = np.full((1, 1, 1), 20.0, np.float32)
    M = np.full((1, 1, 1), 21.0, np.float32)
    u0 = np.float32(value) * np.array([1.0, -0.3, 0.7], np.float32).reshape(3, 1, 1, 1)
    for variant in (0, 1, 2, 5):
        want = _register(dl, S, M, variant, 3, u0, plain_kernels=1)[1]
        got = _register(dl, S, M, variant, 3, u0, **FORMS[form])[1]
        np.testing.assert_array_equal(got, want, err_msg=f"variant {variant}")


@pytest.mark.parametrize("dims", [(8, 8, 4), (40, 32, 24), (129, 128, 60)],
                         ids=["small", "tiles", "strips"])
@pytest.mark.parametrize("value", [1e25, 1e-20], ids=str)
def test_stop_test_at_the_ends_of_the_float_range(dl, dims, value):
    """Equal constant images move nothing, so every norm of the start field is
    met by every iteration: |u|^2 beyond the float range is no convergence and a
    subnormal one is a norm like any other."""
    S = np.full(dims[::-1], 20.0, np.float32)
    u0 = np.full((3,) + dims[::-1], value, np.float32)
    kw = dict(stop_mode=1, eps=1e-6, stop_window=3)
    want = _register(dl, S, S, 0, 9, u0, plain_kernels=1, **kw)
    got = _register(dl, S, S, 0, 9, u0, **kw)
    assert want[0] == (9 if value > 1.0 else 4)
    assert got[0] == want[0]
    assert np.array_equal(np.isnan(got[1]), np.isnan(want[1]))


@pytest.mark.parametrize("dims", [(32, 32, 16), (16, 16, 8), (25, 25, 10)],
                         ids=lambda d: "x".join(map(str, d)))
def test_sum_of_one_large_and_many_small_terms(dl, dims):
    """d = 1 everywhere but 2^15 in one voxel: an FP32 sum that holds 2^30 loses
    every 1 added to it.  The sum of a resident level may lose no more of them than
    the plain kernels', whose FP32 sums end with a warp."""
    n = dims[0] * dims[1] * dims[2]
    exact = float(n - 1) + 2.0 ** 30
    for at in (0, n // 3, n // 2 + 17, n - 1):
        S = np.zeros(dims[::-1], np.float32)
        M = np.ones(dims[::-1], np.float32)
        M.reshape(-1)[at] = 2.0 ** 15
        for variant in (0, 2, 5):
            plain = _register(dl, S, M, variant, 1, plain_kernels=1)[1][0, 0] * n
            level = _register(dl, S, M, variant, 1)[1][0, 0] * n
            assert abs(level - exact) <= abs(plain - exact), (at, variant, exact - plain)


def test_infinite_sum_of_a_resident_level(dl):
    """One difference whose square overflows makes the sum infinite, as in the
    plain kernels, not NaN."""
    S = np.zeros((8, 16, 16), np.float32)
    M = np.ones_like(S)
    M[3, 4, 5] = 1e25
    for variant in (0, 2, 5):
        plain = _register(dl, S, M, variant, 1, plain_kernels=1)[1]
        level = _register(dl, S, M, variant, 1)[1]
        np.testing.assert_array_equal(level[:, 0], plain[:, 0])
        assert np.isinf(plain[0, 0])


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("dims", [(32, 32, 16), (16, 16, 8), (25, 25, 10)],
                         ids=lambda d: "x".join(map(str, d)))
def test_correlation_beside_one_large_term(dl, dims, form):
    """S and M are 1 but for a voxel where S is L, M 0 and another where it is the
    other way round, so that the covariance is what the L^2 in sum S^2 leaves of the
    ones beside it: an FP32 sum of at most 32 voxels loses at most 31 of them."""
    n = dims[0] * dims[1] * dims[2]
    large = 2.0 ** 15
    for at in (5, n // 3):
        S = np.ones(dims[::-1], np.float32)
        M = np.ones(dims[::-1], np.float32)
        S.reshape(-1)[at], M.reshape(-1)[at] = large, 0.0
        S.reshape(-1)[at + n // 2], M.reshape(-1)[at + n // 2] = 0.0, large
        exact = np.corrcoef(S.ravel().astype(np.float64), M.ravel().astype(np.float64))[0, 1]
        for variant in (0, 2, 5):
            p = dl.dir_params_default(levels=1, iters=[1], alpha=0.7, correlation=1,
                                      **FORMS[form])
            ctx = dl.dir_create(S, M, dims, (1.0, 1.0, 1.0), dl.DIR_F32, False, variant, p)
            dl.dir_register(ctx)
            rho = dl.dir_get_correlation(ctx, 1)[0]
            dl.dir_destroy(ctx)
            assert abs(rho - exact) <= 32.0 / (n * float(S.var(dtype=np.float64))), (variant, at)
