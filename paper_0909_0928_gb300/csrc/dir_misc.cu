// dir_misc.cu -- once-per-level and once-per-registration kernels:
// pyramid decimation and field up-sampling (Sec. 2.3), the final warp
// (Sec. 2.5 interpolation), the inverse-consistent output field (Eq. 6), field
// import/export, and the relative-norm stop test (Sec. 2.4).
#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "dir_common.cuh"
#include "dir_launch.h"
#include "dir_pair.cuh"
#include "dir_stop.cuh"

namespace dirk {

constexpr int MTX = 32, MTY = 8;

static dim3 grid_for(const Grid3& g) {
    return dim3((g.nx + MTX - 1) / MTX, (g.ny + MTY - 1) / MTY, g.nz);
}

template <typename Real>
__global__ void decimate_kernel(const Real* __restrict__ in, Grid3 gi, Real* __restrict__ out,
                                Grid3 go) {
    const int x = blockIdx.x * MTX + threadIdx.x, y = blockIdx.y * MTY + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= go.nx || y >= go.ny) return;
    out[offs(go, x, y, z)] = __ldg(in + offs(gi, 2 * x, 2 * y, 2 * z));
}

// fine(x) = 2 * trilinear(coarse, x / 2).  A thread makes the 2 x 2 x 2 fine
// voxels of one coarse cell from its eight corners (24 loads for 24 values; a
// thread per fine voxel gathered 24 per three values: 55.7 us at 256x256x100, now
// 21).
// The lerps and their weights are those of `trilinear`: along each axis the even
// voxel sits on the cell's corner (weight 0) and the odd one half way; past the
// last corner both clamp to it (weight 1 from the corner before).
template <typename Real, typename TF>
__global__ void upsample_kernel(const TF* __restrict__ coarse, Grid3 gc, TF* __restrict__ fine,
                                Grid3 gf) {
    const int X = blockIdx.x * MTX + threadIdx.x, Y = blockIdx.y * MTY + threadIdx.y;
    const int Z = blockIdx.z;
    if (X >= gc.nx || Y >= gc.ny) return;
    auto axis = [](int i, int n, int& i0, int& i1, Real (&f)[2]) {
        const bool last = i >= n - 1;
        i0 = n < 2 ? 0 : (last ? n - 2 : i);
        i1 = n < 2 ? 0 : i0 + 1;
        f[0] = (last && n > 1) ? Real(1) : Real(0);
        f[1] = n < 2 ? Real(0) : (last ? Real(1) : Real(0.5));
    };
    int x0, x1, y0, y1, z0, z1;
    Real fx[2], fy[2], fz[2];
    axis(X, gc.nx, x0, x1, fx);
    axis(Y, gc.ny, y0, y1, fy);
    axis(Z, gc.nz, z0, z1, fz);
    const int r[4] = {offs(gc, 0, y0, z0), offs(gc, 0, y1, z0), offs(gc, 0, y0, z1),
                      offs(gc, 0, y1, z1)};
    const int ofine = offs(gf, 2 * X, 2 * Y, 2 * Z);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const TF* p = coarse + c * gc.cs;
        TF* q = fine + c * gf.cs;
        Real rx[4][2];  // the four rows lerped along x, even and odd
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const Real a = ldg_as<Real>(p + r[k] + x0), b = ldg_as<Real>(p + r[k] + x1);
#pragma unroll
            for (int i = 0; i < 2; ++i) rx[k][i] = r_fma(b, fx[i], a * (Real(1) - fx[i]));
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (2 * Y + j >= gf.ny) break;
            Real v0[2], v1[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                v0[i] = r_fma(rx[1][i], fy[j], rx[0][i] * (Real(1) - fy[j]));
                v1[i] = r_fma(rx[3][i], fy[j], rx[2][i] * (Real(1) - fy[j]));
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (2 * Z + k >= gf.nz) break;
                TF o[2];
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    o[i] = st_as<TF>(Real(2) * r_fma(v1[i], fz[k], v0[i] * (Real(1) - fz[k])));
                TF* d = q + ofine + j * gf.px + k * (int)gf.plane;
                if constexpr (std::is_same<TF, float>::value) {
                    if (2 * X + 1 < gf.nx) {
                        *reinterpret_cast<float2*>(d) = make_float2(o[0], o[1]);
                        continue;
                    }
                }
                d[0] = o[0];
                if (2 * X + 1 < gf.nx) d[1] = o[1];
            }
        }
    }
}

template <typename Real, typename TF>
__global__ void warp_kernel(const Real* __restrict__ img, const TF* __restrict__ u, Grid3 g,
                            float* __restrict__ out) {
    const int x = blockIdx.x * MTX + threadIdx.x, y = blockIdx.y * MTY + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const long long o = (long long)offs(g, x, y, z);
    const Real w = trilinear<Real>(img, g, x, ldg_as<Real>(u + o), y, ldg_as<Real>(u + o + g.cs),
                                   z, ldg_as<Real>(u + o + 2 * g.cs));
    out[(long long)x + (long long)g.nx * ((long long)y + (long long)g.ny * z)] = (float)w;
}

// The same in single precision, two voxels per packed operation and four per
// thread; img with a grid of its own (a dense image: px = nx), at least two
// columns wide (the upper corner of a one-voxel x axis would lie past a dense
// image's last row).  dir_warp at 256x256x100 with a device image: 94 us with a
// pitched copy of it and warp_kernel, now 47.
constexpr int WZ = 4;
__global__ void __launch_bounds__(MTX * MTY)
    warp_pair_kernel(const float* __restrict__ img, Grid3 gi, const float* __restrict__ u, Grid3 g,
                     float* __restrict__ out) {
    const int x = blockIdx.x * MTX + threadIdx.x, y = blockIdx.y * MTY + threadIdx.y;
    const int z = blockIdx.z * WZ;
    if (x >= g.nx || y >= g.ny) return;
    const PairInterp<float> ip(gi, x, y, z);
    const uint32_t o = 4u * (uint32_t)offs(g, x, y, z), pl = 4u * (uint32_t)g.plane;
    const int left = g.nz - z;  // planes from z on
    f32x2 uu[WZ / 2][3];
#pragma unroll
    for (int k = 0; k < WZ / 2; ++k)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            uu[k][c] = f2_pack(__ldg(at_byte(u + c * g.cs, o + min(k, left - 1) * pl)),
                               __ldg(at_byte(u + c * g.cs, o + min(k + WZ / 2, left - 1) * pl)));
    const size_t row = (size_t)g.nx * g.ny;
    float* d = out + x + (size_t)g.nx * y + row * z;
#pragma unroll
    for (int k = 0; k < WZ / 2; ++k) {
        const f32x2 w = ip.at(img, min(k, left - 1), min(k + WZ / 2, left - 1), uu[k][0], uu[k][1],
                              uu[k][2], 0ull);
        if (k < left) d[k * row] = f2_lo(w);
        if (k + WZ / 2 < left) d[(k + WZ / 2) * row] = f2_hi(w);
    }
}

template <typename Real, typename TF>
__global__ void ic_invert_kernel(const TF* __restrict__ h, TF* __restrict__ u, Grid3 g,
                                 int steps) {
    const int x = blockIdx.x * MTX + threadIdx.x, y = blockIdx.y * MTY + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const TF* hx = h;
    const TF* hy = h + g.cs;
    const TF* hz = h + 2 * g.cs;
    // x* = y + a with a = h(x*), iterated from a = 0; once a step returns its
    // input exactly, every later step would too, so the loop may stop there
    Real ax = 0, ay = 0, az = 0;
    for (int s = 0; s < steps; ++s) {
        const Real nx_ = trilinear<Real>(hx, g, x, ax, y, ay, z, az);
        const Real ny_ = trilinear<Real>(hy, g, x, ax, y, ay, z, az);
        const Real nz_ = trilinear<Real>(hz, g, x, ax, y, ay, z, az);
        const bool fixed = (nx_ == ax) && (ny_ == ay) && (nz_ == az);
        ax = nx_;
        ay = ny_;
        az = nz_;
        if (fixed) break;
    }
    const long long o = (long long)offs(g, x, y, z);
    u[o] = st_as<TF>(Real(2) * trilinear<Real>(hx, g, x, ax, y, ay, z, az));
    u[o + g.cs] = st_as<TF>(Real(2) * trilinear<Real>(hy, g, x, ax, y, ay, z, az));
    u[o + 2 * g.cs] = st_as<TF>(Real(2) * trilinear<Real>(hz, g, x, ax, y, ay, z, az));
}

// The same in single precision from an interleaved copy of h, {hx, hy, hz, 0} per
// voxel: a corner is one 16-byte load instead of three loads, its address and
// weights are found once for the three components, x and y are lerped as a packed
// pair, and the corners stay in registers while a stays in their cell (it leaves it
// in the first few steps only).  256x256x100: 1398 us with ic_invert_kernel, 372 +
// 31 for the copy here (520 with the corners loaded at every step), now bound by
// its arithmetic: 78 instructions a step, 76% of the issue rate.
__global__ void interleave_kernel(const float* __restrict__ h, Grid3 g, float4* __restrict__ q) {
    const int x = blockIdx.x * MTX + threadIdx.x, y = blockIdx.y * MTY + threadIdx.y;
    if (x >= g.nx || y >= g.ny) return;
    const int o = offs(g, x, y, blockIdx.z);
    q[o] = make_float4(h[o], h[o + g.cs], h[o + 2 * g.cs], 0.0f);
}

struct Lerp3 {
    f32x2 xy;
    float z;
};
__device__ __forceinline__ Lerp3 lerp3(const Lerp3& a, const Lerp3& b, float f) {
    const float g = 1.0f - f;
    return {f2_fma(b.xy, f2_dup(f), f2_mul(a.xy, f2_dup(g))), fmaf(b.z, f, __fmul_rn(a.z, g))};
}

__global__ void __launch_bounds__(MTX * MTY)
    ic_invert4_kernel(const float4* __restrict__ h, float* __restrict__ u, Grid3 g, int steps) {
    const int x = blockIdx.x * MTX + threadIdx.x, y = blockIdx.y * MTY + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const AxisBounds bx((float)x, g.nx - 1, max(g.nx - 2, 0)),
        by((float)y, g.ny - 1, max(g.ny - 2, 0)), bz((float)z, g.nz - 1, max(g.nz - 2, 0));
    const uint32_t px = 16u * g.px, pl = 16u * (uint32_t)g.plane;
    const uint32_t sx = g.nx > 1 ? 16u : 0u, sy = g.ny > 1 ? px : 0u, sz = g.nz > 1 ? pl : 0u;
    const int o = offs(g, x, y, z);
    const uint32_t o0 = 16u * (uint32_t)o - kMagicBits * (16u + px + pl);
    auto corner = [](float off, const AxisBounds& b, float& f) {  // as pair_corner, one lane
        const float c = r_clamp(off, b.lo, b.hi);
        const float t = fminf(__fadd_rd(c, kMagic), b.top);
        f = c - (t - kMagic);
        return __float_as_uint(t);
    };
    uint32_t held = ~0u;  // byte offset of the cell whose corners c holds (a multiple of 16)
    Lerp3 c[8];
    auto at = [&](float ax, float ay, float az) {  // h at (x, y, z) + a
        float fx, fy, fz;
        const uint32_t p = o0 + 16u * corner(ax, bx, fx) + px * corner(ay, by, fy) +
                           pl * corner(az, bz, fz);
        if (p != held) {
            held = p;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float4 v = __ldg(
                    at_byte(h, p + (k & 1 ? sx : 0u) + (k & 2 ? sy : 0u) + (k & 4 ? sz : 0u)));
                c[k] = Lerp3{f2_pack(v.x, v.y), v.z};
            }
        }
        const Lerp3 v0 = lerp3(lerp3(c[0], c[1], fx), lerp3(c[2], c[3], fx), fy);
        const Lerp3 v1 = lerp3(lerp3(c[4], c[5], fx), lerp3(c[6], c[7], fx), fy);
        return lerp3(v0, v1, fz);
    };
    float ax = 0.0f, ay = 0.0f, az = 0.0f;
    for (int s = 0; s < steps; ++s) {
        const Lerp3 n = at(ax, ay, az);
        const bool fixed = f2_lo(n.xy) == ax && f2_hi(n.xy) == ay && n.z == az;
        ax = f2_lo(n.xy);
        ay = f2_hi(n.xy);
        az = n.z;
        if (fixed) break;
    }
    const Lerp3 r = at(ax, ay, az);
    u[o] = 2.0f * f2_lo(r.xy);
    u[o + g.cs] = 2.0f * f2_hi(r.xy);
    u[o + 2 * g.cs] = 2.0f * r.z;
}

// The three components of a column, or of four adjacent ones with 16-byte loads
// and stores (VEC, where the dense rows are aligned; those of a pitched field
// always are).  The scales come in the arithmetic type.  A field read of
// 256x256x100 took 53 us with double scales converted in every thread, now 38; of
// 250x250x100 52, now 44.
template <typename Real, typename TF, typename Out, bool VEC>
__global__ void export_kernel(const TF* __restrict__ f, Grid3 g, Real sx, Real sy, Real sz,
                              Out* __restrict__ dense) {
    const int x = (VEC ? 4 : 1) * (blockIdx.x * MTX + threadIdx.x);
    const int y = blockIdx.y * MTY + threadIdx.y, z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const size_t n = (size_t)g.nx * g.ny * g.nz;
    const size_t d = (size_t)x + (size_t)g.nx * ((size_t)y + (size_t)g.ny * z);
    const int o = offs(g, x, y, z);
    const Real sc[3] = {sx, sy, sz};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if constexpr (VEC) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(f + c * g.cs + o));
            *reinterpret_cast<float4*>(dense + c * n + d) =
                make_float4(sc[c] * v.x, sc[c] * v.y, sc[c] * v.z, sc[c] * v.w);
        } else {
            dense[c * n + d] = (Out)(sc[c] * ld_as<Real>(f + c * g.cs + o));
        }
    }
}

template <typename Real, typename TF>
__global__ void import_kernel(const float* __restrict__ dense, TF* __restrict__ f, Grid3 g,
                              int ncomp) {
    const int x = blockIdx.x * MTX + threadIdx.x, y = blockIdx.y * MTY + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const long long n = (long long)g.nx * g.ny * g.nz;
    const long long o = (long long)offs(g, x, y, z);
    const long long d = (long long)x + (long long)g.nx * ((long long)y + (long long)g.ny * z);
    for (int c = 0; c < ncomp; ++c) f[o + c * g.cs] = st_as<TF>((Real)dense[d + c * n]);
}

// Dense rows of w words into rows of `pitch` words, the whole volume; a block
// takes PITCH_WORDS consecutive dense words, four per thread in flight.  A pair of
// 256x256x100 float images: 73 us by pitched copies, now 33 (int16: 46, 25).
constexpr unsigned PITCH_WORDS = 1024;
template <typename W>
__global__ void __launch_bounds__(256)
    pitch_rows_kernel(const W* __restrict__ dense, W* __restrict__ pitched, unsigned w,
                      unsigned pitch, unsigned words) {
    const unsigned i0 = blockIdx.x * PITCH_WORDS + threadIdx.x;
    W v[4];
#pragma unroll
    for (unsigned k = 0; k < 4; ++k)
        if (i0 + 256 * k < words) v[k] = __ldg(dense + i0 + 256 * k);
#pragma unroll
    for (unsigned k = 0; k < 4; ++k) {
        const unsigned i = i0 + 256 * k, row = i / w;
        if (i < words) pitched[(size_t)row * pitch + (i - row * w)] = v[k];
    }
}

// One pyramid step (Sec. 2.3) of an image in single precision: the unit Gaussian
// (radius 3) evaluated only where the coarser level samples it, in two kernels:
// the x and y passes at even columns and rows of every plane, then the z pass at
// even planes.  Taps oldest first, fused multiply-adds from zero, as the
// smoothing kernels.  Smoothing the whole image and then sampling it took 27.6 +
// 5.2 us per 256x256x100 image (int16: 37.0 + 5.0), now 17.0 + 5.6.
constexpr int PR = 3;
template <typename TI>
__global__ void __launch_bounds__(MTX * MTY)
    pyramid_xy_kernel(const TI* __restrict__ in, Grid3 gi, float* __restrict__ t, Grid3 go,
                      const Taps taps) {
    constexpr int ROWS = 2 * MTY + 2 * PR - 1;  // fine rows 2 Y0 - 3 .. 2 (Y0 + 7) + 3
    __shared__ float xf[ROWS][MTX];
    const int tx = threadIdx.x, ty = threadIdx.y, z = blockIdx.z;
    const int X = blockIdx.x * MTX + tx, Y0 = blockIdx.y * MTY;
    const TI* plane = in + (size_t)gi.plane * z;
    for (int r = ty; r < ROWS; r += MTY) {
        const TI* row = plane + (size_t)gi.px * clampi(2 * Y0 - PR + r, 0, gi.ny - 1);
        float acc = 0.0f;
#pragma unroll
        for (int k = 0; k < 2 * PR + 1; ++k)
            acc = fmaf(taps.wf[k <= PR ? k : 2 * PR - k],
                       ldg_as<float>(row + clampi(2 * X - PR + k, 0, gi.nx - 1)), acc);
        xf[r][tx] = acc;
    }
    __syncthreads();
    const int Y = Y0 + ty;
    if (X >= go.nx || Y >= go.ny) return;
    float acc = 0.0f;
#pragma unroll
    for (int k = 0; k < 2 * PR + 1; ++k)
        acc = fmaf(taps.wf[k <= PR ? k : 2 * PR - k], xf[2 * ty + k][tx], acc);
    t[(size_t)go.plane * z + (size_t)go.px * Y + X] = acc;
}

__global__ void pyramid_z_kernel(const float* __restrict__ t, int nz, float* __restrict__ out,
                                 Grid3 go, const Taps taps) {
    const int X = blockIdx.x * MTX + threadIdx.x, Y = blockIdx.y * MTY + threadIdx.y;
    const int Z = blockIdx.z;
    if (X >= go.nx || Y >= go.ny) return;
    const float* col = t + (size_t)go.px * Y + X;
    float acc = 0.0f;
#pragma unroll
    for (int k = 0; k < 2 * PR + 1; ++k)
        acc = fmaf(taps.wf[k <= PR ? k : 2 * PR - k],
                   __ldg(col + (size_t)go.plane * clampi(2 * Z - PR + k, 0, nz - 1)), acc);
    out[offs(go, X, Y, Z)] = acc;
}

__global__ void stop_test_kernel(const StopTest q) { stop_test(q, true); }

// Dispatch on (arithmetic, field storage): double/double, float/float,
// float/bf16.  `CALL` sees the types as Real and TF.
#define DIR_DISPATCH_F(fp64, ftype, CALL)                      \
    do {                                                       \
        if (fp64) {                                            \
            if (ftype != kStoreF64) return cudaErrorInvalidValue; \
            using Real = double;                               \
            using TF = double;                                 \
            CALL;                                              \
        } else if (ftype == kStoreBF16) {                      \
            using Real = float;                                \
            using TF = bf16;                                   \
            CALL;                                              \
        } else if (ftype == kStoreF32) {                       \
            using Real = float;                                \
            using TF = float;                                  \
            CALL;                                              \
        } else {                                               \
            return cudaErrorInvalidValue;                      \
        }                                                      \
    } while (0)

cudaError_t launch_decimate(bool fp64, const void* in, const Grid3& gin, void* out,
                            const Grid3& gout, cudaStream_t s) {
    if (fp64)
        decimate_kernel<double><<<grid_for(gout), dim3(MTX, MTY), 0, s>>>(
            static_cast<const double*>(in), gin, static_cast<double*>(out), gout);
    else
        decimate_kernel<float><<<grid_for(gout), dim3(MTX, MTY), 0, s>>>(
            static_cast<const float*>(in), gin, static_cast<float*>(out), gout);
    return cudaGetLastError();
}

cudaError_t launch_upsample(bool fp64, int ftype, const void* coarse, const Grid3& gc, void* fine,
                            const Grid3& gf, cudaStream_t s) {
    DIR_DISPATCH_F(fp64, ftype, (upsample_kernel<Real, TF><<<grid_for(gc), dim3(MTX, MTY), 0, s>>>(
                                    static_cast<const TF*>(coarse), gc, static_cast<TF*>(fine), gf)));
    return cudaGetLastError();
}

cudaError_t launch_warp(bool fp64, int ftype, const void* img, const void* u, const Grid3& g,
                        float* out_dense, cudaStream_t s) {
    DIR_DISPATCH_F(fp64, ftype, (warp_kernel<Real, TF><<<grid_for(g), dim3(MTX, MTY), 0, s>>>(
                                    static_cast<const Real*>(img), static_cast<const TF*>(u), g,
                                    out_dense)));
    return cudaGetLastError();
}

cudaError_t launch_warp_pair(const float* img, const Grid3& gi, const float* u, const Grid3& g,
                             float* out_dense, cudaStream_t s) {
    if (g.nx < 2) return cudaErrorInvalidValue;
    dim3 grid = grid_for(g);
    grid.z = (g.nz + WZ - 1) / WZ;
    warp_pair_kernel<<<grid, dim3(MTX, MTY), 0, s>>>(img, gi, u, g, out_dense);
    return cudaGetLastError();
}

bool ic_invert4_supported(const Grid3& g) { return g.cs < (1LL << 28); }  // 32-bit byte offsets

cudaError_t launch_ic_invert4(const float* h, void* scratch, float* u, const Grid3& g, int steps,
                              cudaStream_t s) {
    if (!ic_invert4_supported(g)) return cudaErrorInvalidValue;
    float4* q = static_cast<float4*>(scratch);
    interleave_kernel<<<grid_for(g), dim3(MTX, MTY), 0, s>>>(h, g, q);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    ic_invert4_kernel<<<grid_for(g), dim3(MTX, MTY), 0, s>>>(q, u, g, steps);
    return cudaGetLastError();
}

bool pitch_rows_supported(const void* dense, int esz) {
    return reinterpret_cast<uintptr_t>(dense) % esz == 0;
}

// Words as wide as the dense rows are aligned to: 16 bytes, or one element (4 or 2)
cudaError_t launch_pitch_rows(const void* dense, void* pitched, const Grid3& g, int esz,
                              cudaStream_t s) {
    if (!pitch_rows_supported(dense, esz)) return cudaErrorInvalidValue;
    const bool wide = ((size_t)g.nx * esz) % 16 == 0 && reinterpret_cast<uintptr_t>(dense) % 16 == 0;
    const unsigned wb = wide ? 16 : esz;
    const unsigned w = (unsigned)((size_t)g.nx * esz / wb), pitch = (unsigned)((size_t)g.px * esz / wb);
    const unsigned words = w * (unsigned)(g.ny * g.nz);  // below 2^30: a field is below 2^31 elements
    const unsigned blocks = (words + PITCH_WORDS - 1) / PITCH_WORDS;
    if (wide)
        pitch_rows_kernel<uint4><<<blocks, 256, 0, s>>>(static_cast<const uint4*>(dense),
                                                        static_cast<uint4*>(pitched), w, pitch, words);
    else if (esz == 4)
        pitch_rows_kernel<uint32_t><<<blocks, 256, 0, s>>>(
            static_cast<const uint32_t*>(dense), static_cast<uint32_t*>(pitched), w, pitch, words);
    else if (esz == 2)
        pitch_rows_kernel<uint16_t><<<blocks, 256, 0, s>>>(
            static_cast<const uint16_t*>(dense), static_cast<uint16_t*>(pitched), w, pitch, words);
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_pyramid(int in_type, const void* in, const Grid3& gin, float* scratch,
                           float* out, const Grid3& gout, const Taps& taps, cudaStream_t s) {
    if (taps.R != PR) return cudaErrorInvalidValue;
    dim3 grid = grid_for(gout);
    grid.z = gin.nz;
    if (in_type == kStoreF32)
        pyramid_xy_kernel<float><<<grid, dim3(MTX, MTY), 0, s>>>(static_cast<const float*>(in), gin,
                                                                 scratch, gout, taps);
    else if (in_type == kStoreI16)
        pyramid_xy_kernel<int16_t><<<grid, dim3(MTX, MTY), 0, s>>>(static_cast<const int16_t*>(in),
                                                                   gin, scratch, gout, taps);
    else
        return cudaErrorInvalidValue;
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    pyramid_z_kernel<<<grid_for(gout), dim3(MTX, MTY), 0, s>>>(scratch, gin.nz, out, gout, taps);
    return cudaGetLastError();
}

cudaError_t launch_ic_invert(bool fp64, int ftype, const void* h, void* u, const Grid3& g,
                             int steps, cudaStream_t s) {
    DIR_DISPATCH_F(fp64, ftype, (ic_invert_kernel<Real, TF><<<grid_for(g), dim3(MTX, MTY), 0, s>>>(
                                    static_cast<const TF*>(h), static_cast<TF*>(u), g, steps)));
    return cudaGetLastError();
}

cudaError_t launch_export_field(bool fp64, int ftype, const void* field, const Grid3& g, double sx,
                                double sy, double sz, void* dense, bool out_fp64, cudaStream_t s) {
    if (!fp64 && ftype == kStoreF32 && !out_fp64 && g.nx % 4 == 0 &&
        reinterpret_cast<uintptr_t>(dense) % 16 == 0) {
        dim3 grid = grid_for(g);
        grid.x = (g.nx + 4 * MTX - 1) / (4 * MTX);
        export_kernel<float, float, float, true><<<grid, dim3(MTX, MTY), 0, s>>>(
            static_cast<const float*>(field), g, (float)sx, (float)sy, (float)sz,
            static_cast<float*>(dense));
    } else if (out_fp64) {
        DIR_DISPATCH_F(fp64, ftype,
                       (export_kernel<Real, TF, double, false><<<grid_for(g), dim3(MTX, MTY), 0, s>>>(
                           static_cast<const TF*>(field), g, (Real)sx, (Real)sy, (Real)sz,
                           static_cast<double*>(dense))));
    } else {
        DIR_DISPATCH_F(fp64, ftype,
                       (export_kernel<Real, TF, float, false><<<grid_for(g), dim3(MTX, MTY), 0, s>>>(
                           static_cast<const TF*>(field), g, (Real)sx, (Real)sy, (Real)sz,
                           static_cast<float*>(dense))));
    }
    return cudaGetLastError();
}

cudaError_t launch_import(bool fp64, int out_type, const float* dense, void* pitched,
                          const Grid3& g, int ncomp, cudaStream_t s) {
    DIR_DISPATCH_F(fp64, out_type, (import_kernel<Real, TF><<<grid_for(g), dim3(MTX, MTY), 0, s>>>(
                                       dense, static_cast<TF*>(pitched), g, ncomp)));
    return cudaGetLastError();
}

// One thread waits, bounded, on an mbarrier that nothing arrives on (the
// failure path of the TMA waits), then records that it gave up.
__global__ void wait_probe_kernel(int* err, unsigned long long limit_ns) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    mbar_init(&bar, 1);
    fence_mbar_init();
    if (!mbar_wait_bounded(&bar, 0, limit_ns)) atomicOr(err, kErrTmaTimeout);
}

cudaError_t launch_wait_probe(int* err, unsigned long long limit_ns, cudaStream_t s) {
    wait_probe_kernel<<<1, 32, 0, s>>>(err, limit_ns);
    return cudaGetLastError();
}

cudaError_t launch_stop_test(const StopTest& q, cudaStream_t s) {
    if (q.red == nullptr) return cudaErrorInvalidValue;
    stop_test_kernel<<<1, 1, 0, s>>>(q);
    return cudaGetLastError();
}

}  // namespace dirk
