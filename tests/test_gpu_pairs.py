"""The production iteration kernels against the plain ones at the sizes where
their tiling can go wrong: single voxels along an axis, one more and one less
than a tile, a brick or a strip, volumes thinner than the filter, and brick
depths that do not divide the volume.  Every kernel rounds each voxel as the
plain-load kernels do, so the fields must be equal, not close.
"""
import numpy as np
import pytest

from phantom.generator import random_volume

pytestmark = pytest.mark.gpu

# (nx, ny, nz): tiles are 32 wide, 8 to 32 rows high, bricks 1 to 8 planes deep
DIMS = [(1, 1, 1), (2, 2, 2), (5, 3, 1), (1, 40, 6), (40, 1, 9), (31, 33, 7), (32, 8, 4),
        (33, 9, 13), (64, 32, 25), (65, 31, 6), (97, 43, 17), (129, 64, 12), (36, 200, 5)]


def _run(dl, S, M, dims, variant, i16, **kw):
    p = dl.dir_params_default(levels=1, iters=[4], alpha=0.7, **kw)
    ctx = dl.dir_create(S, M, dims, (1.0, 1.0, 1.0), dl.DIR_I16 if i16 else dl.DIR_F32, False,
                        variant, p)
    try:
        dl.dir_register(ctx)
        u = np.empty((3,) + dims[::-1], np.float32)
        dl.dir_get_field(ctx, u)
        return u, dl.dir_get_history(ctx, 4)
    finally:
        dl.dir_destroy(ctx)


@pytest.mark.parametrize("dims", DIMS, ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("i16", [False, True], ids=["f32", "i16"])
def test_production_kernels_equal_plain(dims, i16):
    import paper_0909_0928_gb300 as dl

    S = np.round(400.0 * random_volume(dims, 11))
    M = np.round(400.0 * random_volume(dims, 12))
    S, M = (a.astype(np.int16 if i16 else np.float32) for a in (S, M))
    for variant in range(6):
        # float images for the plain reference: whole numbers, so the same values
        ref, href = _run(dl, S.astype(np.float32), M.astype(np.float32), dims, variant, False,
                         plain_kernels=1)
        # by default the whole level in one cluster launch (with and without the
        # correlation sums), then the split kernels (fuse 3: Eqs. 3-6 in one pass)
        for kw in ({}, {"correlation": 1}, {"fuse": 4, "pdl": 0}, {"fuse": 3},
                   {"fuse": 4, "correlation": 1}, {"stop_mode": 1, "eps": 0.0}):
            u, h = _run(dl, S, M, dims, variant, i16, **kw)
            assert np.array_equal(u, ref, equal_nan=True), (variant, kw, np.abs(u - ref).max())
            # sums of n positive terms, rounded in FP32 within a thread and a
            # warp and in FP64 beyond: at most 8 voxels and 32 threads deep
            np.testing.assert_allclose(h, href, rtol=64 * 2.0 ** -24)


@pytest.mark.parametrize("dims", [(2, 2, 2), (33, 9, 13), (40, 1, 9), (1, 9, 9), (97, 40, 1),
                                  (64, 31, 26)], ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("i16", [False, True], ids=["f32", "i16"])
def test_pyramid_and_upsampling(dims, i16):
    """Two and three levels equal the plain kernels' pyramid; the upsampled field
    is twice the trilinear interpolation of its own even voxels (weight 0: the
    coarse values, exactly).  Three lerps of three roundings each, of values up
    to the largest: 9 eps."""
    import paper_0909_0928_gb300 as dl

    S = np.round(400.0 * random_volume(dims, 21)).astype(np.int16 if i16 else np.float32)
    M = np.round(400.0 * random_volume(dims, 22)).astype(S.dtype)

    def run(a, b, dt, **kw):
        p = dl.dir_params_default(alpha=0.7, **kw)
        ctx = dl.dir_create(a, b, dims, (1.0, 1.0, 1.0), dt, False, 5, p)
        try:
            dl.dir_register(ctx)
            u = np.empty((3,) + dims[::-1], np.float32)
            return dl.dir_get_field(ctx, u)
        finally:
            dl.dir_destroy(ctx)

    for levels, iters in ((2, [3, 2]), (3, [2, 1, 2])):
        u = run(S, M, dl.DIR_I16 if i16 else dl.DIR_F32, levels=levels, iters=iters)
        ref = run(S.astype(np.float32), M.astype(np.float32), dl.DIR_F32, levels=levels,
                  iters=iters, plain_kernels=1)
        assert np.array_equal(u, ref, equal_nan=True), np.abs(u - ref).max()

    p = dl.dir_params_default(levels=2, iters=[4, 0], alpha=0.7)
    ctx = dl.dir_create(S, M, dims, (1.0, 1.0, 1.0), dl.DIR_I16 if i16 else dl.DIR_F32, False, 0, p)
    dl.dir_register(ctx)
    f = dl.dir_get_field(ctx, np.empty((3,) + dims[::-1], np.float32)).astype(np.float64)
    dl.dir_destroy(ctx)
    want = f[:, ::2, ::2, ::2]
    for axis, n in ((1, dims[2]), (2, dims[1]), (3, dims[0])):
        pos = np.minimum(np.arange(n) / 2, want.shape[axis] - 1)
        lo = np.floor(pos).astype(int)
        hi = np.minimum(lo + 1, want.shape[axis] - 1)
        w = (pos - lo).reshape([-1 if a == axis else 1 for a in range(4)])
        want = want.take(lo, axis) * (1 - w) + want.take(hi, axis) * w
    assert np.abs(f - want).max() <= 9 * 2.0 ** -24 * np.abs(f).max()


@pytest.mark.parametrize("dims", [(1, 5, 4), (2, 2, 2), (33, 9, 13), (40, 1, 9), (64, 31, 6)],
                         ids=lambda d: "x".join(map(str, d)))
def test_device_inputs_and_outputs(dims):
    """Device images, aligned, off by one element, and warped in place, give what
    host images give; a field read anywhere is the same field."""
    import torch

    import paper_0909_0928_gb300 as dl

    n = dims[0] * dims[1] * dims[2]
    shape = dims[::-1]

    def off(a, by=1):  # the same values from a buffer that starts `by` elements in
        b = torch.empty(n + by, dtype=a.dtype, device="cuda")
        b[by:] = a.flatten()
        return b[by:].view(shape)

    for dt, np_t in ((dl.DIR_F32, np.float32), (dl.DIR_I16, np.int16)):
        S = np.round(400.0 * random_volume(dims, 31)).astype(np_t)
        M = np.round(400.0 * random_volume(dims, 32)).astype(np_t)
        got = []
        for a, b, dev in ((S, M, False), (torch.tensor(S).cuda(), torch.tensor(M).cuda(), True),
                          (off(torch.tensor(S).cuda()), off(torch.tensor(M).cuda()), True)):
            p = dl.dir_params_default(levels=1, iters=[5], alpha=0.7)
            ctx = dl.dir_create(a, b, dims, (1.5, 1.0, 2.0), dt, dev, 0, p)
            dl.dir_register(ctx)
            u = dl.dir_get_field(ctx, np.empty((3,) + shape, np.float32))
            mm = torch.empty(3 * n + 1, device="cuda")
            dl.dir_get_field(ctx, mm[1:], in_mm=True, out_on_device=True)
            u64 = dl.dir_get_field_f64(ctx, np.empty((3,) + shape, np.float64))
            assert np.array_equal(u64, u.astype(np.float64), equal_nan=True)
            scale = np.array([1.5, 1.0, 2.0], np.float32).reshape(3, 1, 1, 1)
            assert np.array_equal(mm[1:].cpu().numpy().reshape(u.shape), u * scale, equal_nan=True)
            img = S.astype(np.float32)
            w = dl.dir_warp(ctx, img, np.empty(shape, np.float32))
            d = torch.tensor(img).cuda()
            for src in (d, off(d), d.clone()):
                out = src if src is not d else torch.empty_like(d)
                dl.dir_warp(ctx, src, out, on_device=True)
                assert np.array_equal(out.cpu().numpy(), w, equal_nan=True)
            got.append((u, w))
            dl.dir_destroy(ctx)
        for u, w in got[1:]:
            assert np.array_equal(u, got[0][0], equal_nan=True)
            assert np.array_equal(w, got[0][1], equal_nan=True)


@pytest.mark.parametrize("nz", [60, 64, 90], ids=["D and u fit", "D fits", "neither fits"])
@pytest.mark.parametrize("variant", [2, 5], ids=["active", "inverse_consistent"])
def test_noalloc_scratch_forms(variant, nz):
    """128 x 128 x nz in 48 MiB: every form of the iteration gives the field of a
    context, whose scratch is its own."""
    import torch

    import paper_0909_0928_gb300 as dl

    dims = (128, 128, nz)
    S, M = (torch.tensor(np.round(400.0 * random_volume(dims, k)).astype(np.float32)).cuda()
            for k in (41, 42))
    p = dl.dir_params_default(levels=1, iters=[3], alpha=0.7)
    out = torch.empty((3,) + dims[::-1], device="cuda")
    dl.dir_register_noalloc(S, M, dims, variant, p, out)
    ctx = dl.dir_create(S, M, dims, (1.0, 1.0, 1.0), dl.DIR_F32, True, variant, p)
    dl.dir_register(ctx)
    want = dl.dir_get_field(ctx, np.empty(out.shape, np.float32))
    dl.dir_destroy(ctx)
    assert np.array_equal(out.cpu().numpy(), want, equal_nan=True)


@pytest.mark.parametrize("dims", [(31, 33, 7), (129, 128, 60)], ids=["tiles", "strips"])
@pytest.mark.parametrize("mode", [1, 2], ids=["norm", "correlation"])
def test_stop_test_in_the_smoothing_kernel(dims, mode):
    """The stop test made by the next x/y kernel ends a level where the test's own
    kernel does (plain kernels), with the same field.  eps lies half way between
    two values of |l(t) - l(t - window)| of a run that does not stop, far from the
    rounding of the sums."""
    import paper_0909_0928_gb300 as dl

    S = np.round(400.0 * random_volume(dims, 51)).astype(np.float32)
    M = np.round(400.0 * random_volume(dims, 52)).astype(np.float32)

    def run(n, **kw):
        p = dl.dir_params_default(levels=1, iters=[n], alpha=0.7, **kw)
        ctx = dl.dir_create(S, M, dims, (1.0, 1.0, 1.0), dl.DIR_F32, False, 0, p)
        try:
            st = dl.dir_register(ctx)
            u = dl.dir_get_field(ctx, np.empty((3,) + dims[::-1], np.float32))
            l = (dl.dir_get_history if mode == 1 else dl.dir_get_correlation)(ctx, n)
            return st.iters_run[0], u, l
        finally:
            dl.dir_destroy(ctx)

    n, w = 12, 2
    l = run(n, correlation=1)[2]
    l = l[1:]  # no |u| before the first update
    l = l[:, 1] / l[:, 2] if mode == 1 else l
    step = np.sort(np.abs(l[w:] - l[:-w]))
    eps = float(step[4] + step[5]) / 2
    kw = dict(stop_mode=mode, eps=eps, stop_window=w)
    a, b = run(n, **kw), run(n, plain_kernels=1, **kw)
    assert a[0] == b[0] and w < a[0] < n
    assert np.array_equal(a[1], b[1], equal_nan=True)
