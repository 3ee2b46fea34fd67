"""Forms of the iteration kernels that only several volumes or large ones reach,
against the plain-load kernels: grouped launches over up to 16 jobs, beside jobs
whose level a cluster holds; strips, deep bricks and the second z pass of u in a
group; strips with remainders along every axis.  Every kernel rounds each voxel as
the plain ones do, so the fields must be equal.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

RESIDENT = 4  # dir_stats.schedule_finest of a level that a cluster holds


@pytest.fixture(scope="module")
def dl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0909_0928_gb300 as dl
    return dl


def _pair(dims, seed, i16):
    g = torch.Generator(device="cuda").manual_seed(seed)
    S, M = (torch.round(400.0 * torch.randn(dims[::-1], generator=g, device="cuda"))
            for _ in range(2))
    return (S.to(torch.int16), M.to(torch.int16)) if i16 else (S, M)


def _context(dl, pair, dims, variant, iters, **kw):
    dt = dl.DIR_I16 if pair[0].dtype == torch.int16 else dl.DIR_F32
    p = dl.dir_params_default(levels=len(iters), iters=iters, alpha=0.7, **kw)
    return dl.dir_create(*pair, dims, (1.0, 1.0, 1.0), dt, True, variant, p)


def _field(dl, ctx, dims):
    return dl.dir_get_field(ctx, np.empty((3,) + dims[::-1], np.float32))


def _plain(dl, pair, dims, variant, iters):
    # float images: whole numbers, so the same values
    ctx = _context(dl, [a.float() for a in pair], dims, variant, iters, plain_kernels=1)
    try:
        dl.dir_register(ctx)
        return _field(dl, ctx, dims)
    finally:
        dl.dir_destroy(ctx)


def _check_batch(dl, sizes, variant, i16, iters, resident):
    pairs = [_pair(d, 70 + k, i16) for k, d in enumerate(sizes)]
    ctxs = [_context(dl, p, d, variant, iters) for p, d in zip(pairs, sizes)]
    batch = None
    try:
        held = [dl.dir_register(c).schedule_finest == RESIDENT for c in ctxs]
        assert held == [k in resident for k in range(len(sizes))]
        batch = dl.dir_batch_create(ctxs)
        assert dl.dir_batch_grouped(batch)
        for k, c in enumerate(ctxs):  # what the registration left is not the answer
            dl.dir_load(c, *pairs[k], dl.DIR_I16 if i16 else dl.DIR_F32, True)
        dl.dir_batch_run(batch)
        for k, (c, p, d) in enumerate(zip(ctxs, pairs, sizes)):
            want = _plain(dl, p, d, variant, iters)
            assert np.array_equal(_field(dl, c, d), want, equal_nan=True), (variant, k, d)
    finally:
        dl.dir_batch_destroy(batch)
        for c in ctxs:
            dl.dir_destroy(c)


@pytest.mark.parametrize("variant", [0, 1, 2, 5])
@pytest.mark.parametrize("small", [(), (0, 6, 7, 15)], ids=["16 in lockstep", "4 resident"])
def test_chunk_of_sixteen(dl, variant, small):
    sizes = [(40 + 3 * (k % 6), 32 + 2 * (k % 5), 20 + k % 7) for k in range(16)]
    for k in small:
        sizes[k] = (20 + k, 18, 11)
    _check_batch(dl, sizes, variant, variant == 1, [4, 3], small)


# three volumes of (608, 912] four-plane bricks, just over a wave of resident ones:
# six-plane bricks for Eq. 1, eight-plane ones for Eq. 2; and above 2^20 voxels and
# 16 strips per SM: strips, and u of Eqs. 3-6 formed again by the force kernel
GROUPS = {"deep bricks": [(96, 64, 48), (90, 61, 47), (95, 63, 46)],
          "strips": [(97, 83, 45), (64, 90, 50), (101, 77, 47), (96, 85, 43), (89, 86, 49),
                     (100, 80, 41)]}


@pytest.mark.parametrize("variant", range(6))
@pytest.mark.parametrize("sizes", list(GROUPS))
@pytest.mark.parametrize("i16", [False, True], ids=["f32", "i16"])
def test_large_chunks(dl, sizes, variant, i16):
    _check_batch(dl, GROUPS[sizes], variant, i16, [3], ())


@pytest.mark.parametrize("graph", [1, 0], ids=["graph", "direct"])
@pytest.mark.parametrize("variant", [0, 1, 2, 5])
@pytest.mark.parametrize("dims", [(193, 171, 87), (161, 149, 49), (129, 127, 61), (260, 50, 70)],
                         ids=lambda d: "x".join(map(str, d)))
def test_strips_with_remainders(dl, dims, variant, graph):
    pair = _pair(dims, 90, variant == 1)
    # launched directly the kernels start before the one before them has ended
    ctx = _context(dl, pair, dims, variant, [6], use_graph=graph)
    try:
        dl.dir_register(ctx)
        got = _field(dl, ctx, dims)
    finally:
        dl.dir_destroy(ctx)
    assert np.array_equal(got, _plain(dl, pair, dims, variant, [6]), equal_nan=True)
