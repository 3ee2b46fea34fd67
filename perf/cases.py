"""Performance cases of the registration library: what its users have it do.

A case is one pass through the public Python binding: a registration of a new
image pair on a resident context (dir_load, dir_register, dir_get_field, and
dir_warp where the deformed image is wanted), a batch of registrations, a
registration without device allocation, or the use of a registered field.
Images are synthetic chest-like CT pairs in HU: a body and two lungs with soft
edges, vessels, 20 HU of noise drawn separately for both images, and a smooth
respiratory deformation of a few voxels.

Each case names its kind ("register", "batch", "noalloc", "apply"), the volume
size, the force law, the pyramid's depth and iterations (coarsest first), the
storage of the images and the options it takes.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_0909_0928_gb300 as dl

SPACING = (0.9, 0.9, 2.5)  # mm per voxel


def _case(name, kind, dims, variant, iters, **more):
    c = {"name": name, "kind": kind, "nx": dims[0], "ny": dims[1], "nz": dims[2],
         "variant": variant, "iters": iters, "alpha": 0.4, "int16": False, "host": False,
         "warp": False, "stop": False, "init": False, "pairs": 1}
    c.update(more)
    return c


def listed():
    return [
        # the smallest volume the library is used on (cropped region, thumbnail
        # alignment): hundreds of tiny launches, so latency and launch gaps
        _case("small_passive", "register", (64, 64, 32), "passive", "200/100/50"),
        # the standard case: one clinical thoracic pair, the default schedule,
        # with the deformed image for review
        _case("ct_passive", "register", (256, 256, 100), "passive", "200/100/50", warp=True),
        # the same from scanner storage: int16 HU in pinned host memory, the
        # field returned to the host; the evolved passive law reads grad M too
        _case("ct_evolved_host", "register", (256, 256, 100), "evolved_passive", "200/100/50",
              int16=True, host=True),
        # the laws that need the gradient of the warped image
        _case("ct_active", "register", (256, 256, 100), "active", "200/100/50"),
        # the inverse-consistent law: both images warped every iteration
        _case("ct_inverse", "register", (256, 256, 100), "inverse_consistent", "200/100/50"),
        # an odd, cropped volume and the paper's own two levels
        _case("ragged_double", "register", (193, 171, 87), "double", "60/30"),
        # the largest volume of the serving mix (whole chest, thin slices)
        _case("chest_adjusted", "register", (512, 512, 160), "adjusted_double", "200/100/50",
              alpha=2.0, int16=True),
        # the schedule as an upper bound with the relative-norm stop test
        _case("ct_stop", "register", (256, 256, 100), "passive", "200/100/50", stop=True),
        # refinement of a field already at hand on one level
        _case("refine", "register", (192, 160, 96), "passive", "20", init=True),
        # many small pairs at once (regions of interest of one study)
        _case("batch_rois", "batch", (64, 64, 32), "passive", "200/100/50", pairs=16, int16=True),
        # a host that owns the device's memory: no allocation, direct launches
        _case("noalloc_active", "noalloc", (128, 128, 64), "active", "200/100/50"),
        # a registered field put to use: another image warped, the field in mm
        _case("apply_field", "apply", (256, 256, 100), "passive", "20/10/5"),
    ]


def draw(rng):
    c = _draw(rng)
    del c["name"]
    return c


def _draw(rng):
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n if rng.random() < 0.5 else max(lo, n // 16 * 16)

    law = rng.choice(["passive", "evolved_passive", "active", "double", "adjusted_double",
                      "inverse_consistent"])
    alpha = rng.choice([0.4, 2.0])
    int16 = rng.random() < 0.4
    f = rng.choice([1, 1, 2, 4])  # full, half and quarter schedules
    iters = rng.choice(["200/100/50", "100/50", "200/100/50"])
    iters = "/".join(str(int(k) // f) for k in iters.split("/"))
    kind = rng.choice(["register"] * 7 + ["batch", "noalloc", "apply"])
    if kind == "batch":
        dims = (size(48, 128), size(48, 128), size(24, 64))
        return _case("", kind, dims, law, iters, alpha=alpha, int16=int16,
                     pairs=rng.choice([4, 8, 16]))
    if kind == "noalloc":
        dims = (size(48, 128), size(48, 128), size(24, 64))
        return _case("", kind, dims, law, iters, alpha=alpha)
    dims = (size(48, 384), size(48, 384), size(24, 128))
    if kind == "apply":
        return _case("", kind, dims, law, "20/10/5", alpha=alpha)
    opt = rng.choice(["", "", "", "warp", "host", "stop", "init"])
    more = {opt: True} if opt else {}
    if opt == "init":
        iters = str(rng.randint(5, 40))
    return _case("", kind, dims, law, iters, alpha=alpha, int16=int16, **more)


# ------------------------------------------------------------------- inputs

def _grid(n, device):
    return torch.arange(n, dtype=torch.float32, device=device)


def _sizes(case):
    """The volume sizes of a case: one, or the uneven sizes of a batch."""
    n = (case["nx"], case["ny"], case["nz"])
    if case["kind"] != "batch":
        return [n]
    # regions of interest differ by up to a quarter per axis
    r = random.Random(n[0] * 1009 + n[1] * 31 + n[2])
    return [n] + [tuple(int(a * r.uniform(0.75, 1.0)) for a in n) for _ in range(case["pairs"] - 1)]


def _deformation(dims, rng, device):
    """A smooth backward map in voxels: Gaussian bumps and a stretch along z."""
    nx, ny, nz = dims
    axes = [_grid(n, device) for n in dims]
    scale = 0.04 * min(nx, ny)
    v = [torch.zeros((nz, ny, nx), device=device) for _ in range(3)]
    for _ in range(6):
        c = [rng.uniform(0.25, 0.75) * n for n in dims]
        w = [rng.uniform(0.10, 0.20) * n for n in dims]
        e = [torch.exp(-0.5 * ((a - ci) / wi) ** 2) for a, ci, wi in zip(axes, c, w)]
        bump = e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :]
        d = [rng.gauss(0.0, 1.0) for _ in range(3)]
        s = rng.uniform(0.4, 0.9) * scale / math.sqrt(sum(t * t for t in d))
        for comp in range(3):
            v[comp] += (s * d[comp] * (0.4 if comp == 2 else 1.0)) * bump
    v[2] += rng.uniform(0.05, 0.10) * torch.clamp(0.5 * nz - axes[2], min=0.0)[:, None, None]
    return v


def _anatomy(dims, rng):
    lungs = [(0.30 + rng.uniform(-0.02, 0.02), 0.5, 0.5), (0.70 + rng.uniform(-0.02, 0.02), 0.5, 0.5)]
    tubes = []
    for _ in range(24):
        c = lungs[rng.randint(0, 1)]
        a = [(ci + rng.uniform(-s, s)) * (n - 1)
             for ci, s, n in zip(c, (0.10, 0.18, 0.30), dims)]
        b = [ai + rng.uniform(-0.16, 0.16) * n for ai, n in zip(a, dims)]
        tubes.append((a, b, rng.uniform(1.0, 3.0)))
    return lungs, tubes


def _image(dims, anatomy, p):
    """HU at the positions p = [px, py, pz] (tensors that broadcast to a volume)."""
    nx, ny, nz = dims

    def inside(c, half):
        q = sum(((pi - ci * (n - 1)) / (h * n)) ** 2 for pi, ci, h, n in zip(p, c, half, dims))
        return torch.sigmoid((1.0 - torch.sqrt(q + 1e-6)) * (0.6 * min(h * n for h, n in zip(half, dims))))

    lungs, tubes = anatomy
    body = inside((0.5, 0.5, 0.5), (0.46, 0.38, 0.60))
    lung = torch.maximum(inside(lungs[0], (0.16, 0.26, 0.42)), inside(lungs[1], (0.16, 0.26, 0.42)))
    img = -1000.0 + 1000.0 * body
    img = img + lung * (-850.0 - img)
    vessel = torch.zeros_like(img)
    for a, b, r in tubes:
        ab = [bi - ai for ai, bi in zip(a, b)]
        t = sum((pi - ai) * d for pi, ai, d in zip(p, a, ab)) / max(sum(d * d for d in ab), 1e-3)
        t = torch.clamp(t, 0.0, 1.0)
        d2 = sum((pi - ai - t * d) ** 2 for pi, ai, d in zip(p, a, ab))
        vessel = torch.maximum(vessel, torch.sigmoid(2.0 * (r - torch.sqrt(d2 + 1e-6))))
    return img + (vessel * lung) * (40.0 - img)


def _pair(dims, seed, int16):
    """Static and moving volume of shape (nz, ny, nx) on the GPU."""
    nx, ny, nz = dims
    device = torch.device("cuda")
    rng = random.Random(seed * 7919 + nx * 131 + ny * 17 + nz)
    anatomy = _anatomy(dims, rng)
    v = _deformation(dims, rng, device)
    x, y, z = (_grid(n, device) for n in dims)
    p = [x[None, None, :], y[None, :, None], z[:, None, None]]
    gen = torch.Generator(device=device).manual_seed(rng.randrange(1 << 30))
    out = []
    for moving in (False, True):
        img = _image(dims, anatomy, [pi + vi for pi, vi in zip(p, v)] if moving else p)
        img = img.expand(nz, ny, nx) + 20.0 * torch.randn((nz, ny, nx), generator=gen, device=device)
        out.append(torch.round(img).to(torch.int16) if int16 else img.contiguous())
    return out


def _start_field(dims, seed):
    """A field at hand before a refinement: a smooth one of about a voxel."""
    v = torch.stack(_deformation(dims, random.Random(seed * 31 + 5), torch.device("cuda")))
    return (v * (1.0 / (0.04 * min(dims[0], dims[1])))).contiguous()


def _iters(case):
    return [int(k) for k in case["iters"].split("/")]


# --------------------------------------------------------------------- runs

class _Job:
    """A resident context, its image pair and the buffers its results go to."""

    def __init__(self, case, dims, seed):
        self.case, self.dims = case, dims
        nx, ny, nz = dims
        self.S, self.M = _pair(dims, seed, case["int16"])
        self.init = _start_field(dims, seed) if case["init"] else None
        it = _iters(case)
        self.params = dl.dir_params_default(levels=len(it), iters=it, alpha=case["alpha"],
                                            stop_mode=1 if case["stop"] else 0,
                                            init_field=self.init)
        self.dtype = dl.DIR_I16 if case["int16"] else dl.DIR_F32
        self.law = dl.VARIANTS[case["variant"]]
        self.ctx = None
        if case["host"]:
            self.S, self.M = self.S.cpu().pin_memory().numpy(), self.M.cpu().pin_memory().numpy()
            self.field = torch.empty((3, nz, ny, nx), pin_memory=True).numpy()
        else:
            self.field = torch.empty((3, nz, ny, nx), device="cuda")
        self.warped = None
        if case["warp"] or case["kind"] == "apply":
            self.warped = torch.empty((nz, ny, nx), device="cuda")
        if case["kind"] != "noalloc":
            self.ctx = dl.dir_create(self.S, self.M, dims, SPACING, self.dtype, not case["host"],
                                     self.law, self.params)

    def load(self):
        dl.dir_load(self.ctx, self.S, self.M, self.dtype, not self.case["host"])

    def read(self, in_mm=False):
        return dl.dir_get_field(self.ctx, self.field, in_mm, not self.case["host"])

    def warp(self):
        image = self.M.float() if self.case["int16"] else self.M
        return dl.dir_warp(self.ctx, image, self.warped, dl.DIR_F32, True)

    def __del__(self):
        if getattr(self, "ctx", None) is not None:
            dl.dir_destroy(self.ctx)
            self.ctx = None


class _Batch:
    def __init__(self, case, seed):
        self.jobs = [_Job(case, d, seed + 100 * k) for k, d in enumerate(_sizes(case))]
        self.batch = dl.dir_batch_create([j.ctx for j in self.jobs])

    def __del__(self):
        if getattr(self, "batch", None) is not None:
            dl.dir_batch_destroy(self.batch)
            self.batch = None


def prepare(case, seed):
    if case["kind"] == "batch":
        return _Batch(case, seed)
    job = _Job(case, _sizes(case)[0], seed)
    if case["kind"] == "apply":
        dl.dir_register(job.ctx)
    return job


def run(state):
    if isinstance(state, _Batch):
        for job in state.jobs:
            job.load()
        dl.dir_batch_run(state.batch)
        return [job.read() for job in state.jobs]
    kind = state.case["kind"]
    if kind == "noalloc":
        dl.dir_register_noalloc(state.S, state.M, state.dims, state.law, state.params, state.field)
        return [state.field]
    if kind == "apply":
        return [state.warp(), state.read(in_mm=True)]
    state.load()
    dl.dir_register(state.ctx)
    out = [state.read()]
    if state.warped is not None:
        out.append(state.warp())
    return out


# --------------------------------------------------------------------- work

def _level_sizes(dims, levels):
    out = [tuple(dims)]
    for _ in range(1, levels):
        out.append(tuple((n + 1) // 2 for n in out[-1]))
    return out


def work(case):
    """Every iteration reads the field and both images of its level and writes
    the field (12 + 12 bytes and two voxels), whatever the kernels in between
    keep on the chip; the images come in and the field goes out once.  Per
    voxel-update: 63 fused multiply-adds of the Gaussian, 29 operations of a
    trilinear interpolation, 9 of a gradient, 20 of a force and update."""
    esz = 2 if case["int16"] else 4
    it = _iters(case)
    ops = 126 + 29 + 9 + 20
    if case["variant"] not in ("passive",):
        ops += 9
    if case["variant"] in ("double", "adjusted_double"):
        ops += 12
    if case["variant"] == "inverse_consistent":
        ops += 29
    total_b = total_f = 0
    for dims in _sizes(case):
        n = dims[0] * dims[1] * dims[2]
        if case["kind"] == "apply":  # field and image in, warped image and field out
            total_b += n * (12 + 4 + 4 + 12)
            total_f += n * 32
            continue
        total_b += n * (2 * esz + 12)
        for lc, d in enumerate(reversed(_level_sizes(dims, len(it)))):
            k = it[lc] if not case["stop"] else min(it[lc], 14)  # it stops after 10 and a few
            m = d[0] * d[1] * d[2]
            total_b += m * k * (24 + 2 * (esz if lc == len(it) - 1 else 4))
            total_f += m * k * ops
        if case["warp"]:
            total_b += n * (12 + 4 + 4)
            total_f += n * 29
    return {"bytes": total_b, "flops": total_f}


# ---------------------------------------------------- 64-bit reference values

def _taps(sigma=1.0):
    r = math.ceil(3 * sigma)
    w = [math.exp(-t * t / (2.0 * sigma * sigma)) for t in range(-r, r + 1)]
    return [t / sum(w) for t in w]


def _smooth(a):
    """Gaussian of unit deviation along x, y, z of (..., nz, ny, nx), edges replicated."""
    w = _taps()
    r = len(w) // 2
    for dim in (-1, -2, -3):
        n = a.shape[dim]
        first, last = a.narrow(dim, 0, 1), a.narrow(dim, n - 1, 1)
        p = torch.cat([first] * r + [a] + [last] * r, dim)
        a = w[0] * p.narrow(dim, 0, n)
        for t in range(1, len(w)):
            a.add_(p.narrow(dim, t, n), alpha=w[t])
    return a


def _gradient(a):
    out = []
    for dim in (2, 1, 0):
        n = a.shape[dim]
        p = torch.cat([a.narrow(dim, 0, 1), a, a.narrow(dim, n - 1, 1)], dim)
        out.append(0.5 * (p.narrow(dim, 2, n) - p.narrow(dim, 0, n)))
    return out


def _sample(vols, pos):
    """Trilinear values of volumes of one shape at pos = [x, y, z], coordinates clamped."""
    nz, ny, nx = vols[0].shape
    base, fr, up = 0, [], []
    for p, n, stride in zip(pos, (nx, ny, nz), (1, nx, nx * ny)):
        p = p.clamp(0.0, n - 1.0)
        i = p.floor().clamp(max=max(n - 2, 0))
        fr.append(p - i)
        up.append(stride if n > 1 else 0)
        base = base + i.long() * stride
    out = []
    for v in vols:
        f = v.reshape(-1)
        planes = []
        for oz in (0, up[2]):
            rows = [torch.lerp(f[base + (oz + oy)], f[base + (oz + oy + up[0])], fr[0])
                    for oy in (0, up[1])]
            planes.append(torch.lerp(rows[0], rows[1], fr[1]))
        out.append(torch.lerp(planes[0], planes[1], fr[2]))
    return out


def _points(shape, device):
    nz, ny, nx = shape
    g = [torch.arange(n, dtype=torch.float64, device=device) for n in (nx, ny, nz)]
    return [g[0][None, None, :].expand(shape), g[1][None, :, None].expand(shape),
            g[2][:, None, None].expand(shape)]


def _quotient(d, den):
    return torch.where(den == 0.0, torch.zeros_like(d), d / den)


def _sum_sq(g):
    return g[0] * g[0] + g[1] * g[1] + g[2] * g[2]


def _register64(S, M, case):
    """The registration in double precision: field (3, nz, ny, nx) in voxels."""
    it = _iters(case)
    law = case["variant"]
    pyr = [(S.double(), M.double())]
    for _ in range(1, len(it)):
        pyr.append(tuple(_smooth(a)[::2, ::2, ::2].contiguous() for a in pyr[-1]))
    u = None
    for lc, k in enumerate(it):
        S, M = pyr[len(it) - 1 - lc]
        pts = _points(S.shape, S.device)
        if u is None:
            u = torch.zeros((3,) + tuple(S.shape), dtype=torch.float64, device=S.device)
            if case["init"]:
                u = case["start"].double()
        else:
            u = 2.0 * torch.stack(_sample([u[0], u[1], u[2]], [0.5 * p for p in pts]))
        gs = _gradient(S)
        if law == "evolved_passive":
            b = torch.sqrt(_sum_sq(_gradient(M)))
        history = []
        for n in range(k):
            W = _sample([M], [p + c for p, c in zip(pts, u)])[0]
            d = W - S
            if law == "passive":
                q = _quotient(d, d * d + _sum_sq(gs))
                du = [-q * g for g in gs]
            elif law == "evolved_passive":
                a2 = _sum_sq(gs)
                s = a2 + b * b
                q = _quotient(4.0 * d * torch.sqrt(a2) * b, (2.0 * d * d + s) * s)
                du = [-q * g for g in gs]
            elif law == "inverse_consistent":
                Ws = _sample([S], [p - c for p, c in zip(pts, u)])[0]
                d = W - Ws
                gm = _gradient(W + Ws)
                q = _quotient(d, d * d + _sum_sq(gm))
                du = [-q * g for g in gm]
            else:
                gm = _gradient(W)
                c = case["alpha"] ** 2 if law == "adjusted_double" else 1.0
                q = _quotient(d, c * d * d + _sum_sq(gm))
                du = [-q * g for g in gm]
                if law != "active":
                    q = _quotient(d, c * d * d + _sum_sq(gs))
                    du = [a - q * g for a, g in zip(du, gs)]
            if case["stop"]:
                total = float(torch.sqrt(_sum_sq(u)).sum())
                step = float(torch.sqrt(_sum_sq(du)).sum())
                history.append(step / total if total > 0.0 else math.nan)
            u = _smooth(u + torch.stack(du))
            if case["stop"] and n >= 10 and abs(history[n] - history[n - 10]) <= 1e-4:
                break
    if law == "inverse_consistent":  # the static-grid field of the mid-space field
        pts = _points(u.shape[1:], u.device)
        h = [u[0], u[1], u[2]]
        pos = pts
        for _ in range(20):
            pos = [p + a for p, a in zip(pts, _sample(h, pos))]
        u = 2.0 * torch.stack(_sample(h, pos))
    return u


def exact(case, seed):
    fields, warped = [], []
    for k, dims in enumerate(_sizes(case)):
        s = seed + 100 * k if case["kind"] == "batch" else seed
        S, M = _pair(dims, s, case["int16"])
        u = _register64(S, M, dict(case, start=_start_field(dims, s)))
        if case["warp"] or case["kind"] == "apply":
            pts = _points(S.shape, S.device)
            warped.append(_sample([M.double()], [p + c for p, c in zip(pts, u)])[0])
        if case["kind"] == "apply":
            u = u * torch.tensor(SPACING, dtype=torch.float64, device=u.device)[:, None, None, None]
        fields.append(u.cpu().numpy() if case["host"] else u)
    if case["kind"] == "apply":
        return [warped[0], fields[0]]
    return fields + warped
