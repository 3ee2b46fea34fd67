// dir_pair.cuh -- two voxels at a time: the per-voxel work of a single-precision
// demons iteration (Sec. 2.5 interpolation, Eqs. (1)-(6)) on the two lanes of
// the packed f32x2 instructions.
//
// A thread owns a z column of its brick and pairs voxel k with voxel
// k + FTZ/2, so that both lanes of every operand come from loads of their own
// and no register moves are needed to build a pair.  Every packed operation
// rounds each lane exactly as the scalar one in dir_force_kernel.cuh and
// dir_force_law.cuh would, so a kernel built from these gives the same field
// bit for bit.  The split kernels are bound by instruction issue, not by
// memory (256x256x100: the z + force kernel issued 242 warp instructions per
// 32 voxels with scalar arithmetic), which is what the pairing halves.
#pragma once

#include <cuda_runtime.h>

#include "dir_common.cuh"
#include "dir_force_kernel.cuh"

namespace dirk {

__device__ __forceinline__ f32x2 f2_sub(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 f2_add_rm(f32x2 a, f32x2 b) {  // rounds toward -inf
    f32x2 d;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 f2_dup(float a) { return f2_pack(a, a); }
__device__ __forceinline__ float f2_lo(f32x2 v) {
    float a, b;
    f2_unpack(v, a, b);
    return a;
}
__device__ __forceinline__ float f2_hi(f32x2 v) {
    float a, b;
    f2_unpack(v, a, b);
    return b;
}
// a + b and a - b where an operand is a product that has to be rounded first.
// Done per lane: the assembler merges a packed product with a packed addition
// into one multiply-add, .rn on both or not, which it does not do to the
// scalar instructions.
__device__ __forceinline__ f32x2 f2_add_rounded(f32x2 a, f32x2 b) {
    return f2_pack(__fadd_rn(f2_lo(a), f2_lo(b)), __fadd_rn(f2_hi(a), f2_hi(b)));
}
__device__ __forceinline__ f32x2 f2_sub_rounded(f32x2 a, f32x2 b) {
    return f2_pack(__fsub_rn(f2_lo(a), f2_lo(b)), __fsub_rn(f2_hi(a), f2_hi(b)));
}
__device__ __forceinline__ f32x2 f2_neg(f32x2 a) { return f2_pack(-f2_lo(a), -f2_hi(a)); }
// (x x + y y) + z z with the two additions fused, as r_sq3
__device__ __forceinline__ f32x2 f2_sq3(f32x2 x, f32x2 y, f32x2 z) {
    return f2_fma(z, z, f2_fma(y, y, f2_mul(x, x)));
}
// x x + y y + z z as the compiler contracts it in the scalar kernels: y y rounded
__device__ __forceinline__ f32x2 f2_sq3_yxz(f32x2 x, f32x2 y, f32x2 z) {
    return f2_fma(z, z, f2_fma(x, x, f2_mul(y, y)));
}
// |grad M| of Eq. (2)
__device__ __forceinline__ f32x2 f2_norm_yxz(f32x2 x, f32x2 y, f32x2 z) {
    const f32x2 s = f2_sq3_yxz(x, y, z);
    return f2_pack(r_sqrt(f2_lo(s)), r_sqrt(f2_hi(s)));
}

// 1.5 * 2^23: a float of this size has a unit ulp, so c + kMagic rounded toward
// -inf is kMagic + floor(c) for |c| < 2^22, with the integer in the low bits
// of the word (one packed add instead of a rounding and a conversion per lane,
// both of which run at a quarter of the rate)
constexpr float kMagic = 12582912.0f;
constexpr uint32_t kMagicBits = 0x4b400000u;

// An image value as the arithmetic takes it: a float as it is; an int16 as
// kMagic + value, exact, by an integer add instead of a conversion.  Every use
// is a difference of two image values, which is exact either way and the same.
__device__ __forceinline__ float img_bits(float v) { return v; }
__device__ __forceinline__ float img_bits(int16_t v) {
    return __uint_as_float(kMagicBits + (uint32_t)(int)v);
}
template <typename TI>
__device__ __forceinline__ float img_value(float b) {  // back to the value itself
    return sizeof(TI) == 2 ? b - kMagic : b;
}
// The element at a byte offset of an image: one 32-bit register beside the
// uniform base pointer (an image is below 2^32 bytes: the engine bounds a
// field's three components below 2^31 elements)
template <typename TI>
__device__ __forceinline__ float img_ldg(const TI* base, uint32_t byte) {
    return img_bits(__ldg(reinterpret_cast<const TI*>(reinterpret_cast<const char*>(base) + byte)));
}
template <typename T>
__device__ __forceinline__ T* at_byte(T* base, uint32_t byte) {
    return reinterpret_cast<T*>(reinterpret_cast<char*>(base) + byte);
}
template <typename T>
__device__ __forceinline__ const T* at_byte(const T* base, uint32_t byte) {
    return reinterpret_cast<const T*>(reinterpret_cast<const char*>(base) + byte);
}

// Corner search along one axis for a pair of voxels, bounds as floats: p is
// clamped to [0, n - 1] in offset form (lo = -base, hi = n - 1 - base), its
// floor kept at n - 2 at most (top = kMagic + max(n - 2, 0) - base), the
// weight is what is left: ax_corner's values, lane by lane.
struct AxisBounds {
    float lo, hi, top;
    __device__ __forceinline__ AxisBounds(float base, int nm1, int nm2)
        : lo(-base), hi((float)nm1 - base), top((float)nm2 - base + kMagic) {}
    // of the position k further along the axis (small integers: exact)
    __device__ __forceinline__ AxisBounds(const AxisBounds& b, int k)
        : lo(b.lo - (float)k), hi(b.hi - (float)k), top(b.top - (float)k) {}
};
struct PairCorner {
    uint32_t a, b;  // kMagicBits + (corner - base) of the two lanes
    f32x2 f;        // weights
};
__device__ __forceinline__ PairCorner pair_corner(f32x2 off, const AxisBounds& A,
                                                  const AxisBounds& B) {
    float oa, ob;
    f2_unpack(off, oa, ob);
    const f32x2 c = f2_pack(r_clamp(oa, A.lo, A.hi), r_clamp(ob, B.lo, B.hi));
    float ta, tb;
    f2_unpack(f2_add_rm(c, f2_dup(kMagic)), ta, tb);
    ta = fminf(ta, A.top);
    tb = fminf(tb, B.top);
    PairCorner r;
    r.a = __float_as_uint(ta);
    r.b = __float_as_uint(tb);
    r.f = f2_sub(c, f2_sub(f2_pack(ta, tb), f2_dup(kMagic)));
    return r;
}

// The warped image relative to a reference at two voxels of one column:
// I((x, y, z) + u) - ref, interp_rel lane by lane.
template <typename TI>
struct PairInterp {
    AxisBounds bx, by, bz;       // bz: of the column's first voxel
    uint32_t px, pl, sy, sz;     // bytes: row and plane pitch, steps to the upper corners
    uint32_t o0;                 // byte offset of the column's first voxel, less the bias of
                                 // three kMagicBits-based corners
    __device__ __forceinline__ PairInterp(const Grid3& g, int x, int y, int z)
        : bx((float)x, g.nx - 1, max(g.nx - 2, 0)), by((float)y, g.ny - 1, max(g.ny - 2, 0)),
          bz((float)z, g.nz - 1, max(g.nz - 2, 0)), px((uint32_t)sizeof(TI) * g.px),
          pl((uint32_t)sizeof(TI) * (uint32_t)g.plane), sy(g.ny > 1 ? px : 0), sz(g.nz > 1 ? pl : 0) {
        o0 = (uint32_t)sizeof(TI) * (uint32_t)offs(g, x, y, z) -
             kMagicBits * ((uint32_t)sizeof(TI) + px + pl);
    }
    // the voxels ka and kb above the column's first; ref in img_bits form
    __device__ __forceinline__ f32x2 at(const TI* __restrict__ I, int ka, int kb, const f32x2 ux,
                                        f32x2 uy, f32x2 uz, f32x2 ref) const {
        const PairCorner cx = pair_corner(ux, bx, bx);
        const PairCorner cy = pair_corner(uy, by, by);
        const PairCorner cz = pair_corner(uz, AxisBounds(bz, ka), AxisBounds(bz, kb));
        // lower corners, their rows one further along y, z and both
        const uint32_t a0 = o0 + ka * pl + (uint32_t)sizeof(TI) * cx.a + px * cy.a + pl * cz.a;
        const uint32_t b0 = o0 + kb * pl + (uint32_t)sizeof(TI) * cx.b + px * cy.b + pl * cz.b;
        const uint32_t a1 = a0 + sy, a2 = a0 + sz, a3 = a2 + sy;
        const uint32_t b1 = b0 + sy, b2 = b0 + sz, b3 = b2 + sy;
        const TI* J = I + 1;
        const f32x2 c000 = f2_sub(f2_pack(img_ldg(I, a0), img_ldg(I, b0)), ref);
        const f32x2 c100 = f2_sub(f2_pack(img_ldg(J, a0), img_ldg(J, b0)), ref);
        const f32x2 c010 = f2_sub(f2_pack(img_ldg(I, a1), img_ldg(I, b1)), ref);
        const f32x2 c110 = f2_sub(f2_pack(img_ldg(J, a1), img_ldg(J, b1)), ref);
        const f32x2 c001 = f2_sub(f2_pack(img_ldg(I, a2), img_ldg(I, b2)), ref);
        const f32x2 c101 = f2_sub(f2_pack(img_ldg(J, a2), img_ldg(J, b2)), ref);
        const f32x2 c011 = f2_sub(f2_pack(img_ldg(I, a3), img_ldg(I, b3)), ref);
        const f32x2 c111 = f2_sub(f2_pack(img_ldg(J, a3), img_ldg(J, b3)), ref);
        const f32x2 one = f2_dup(1.0f);
        const f32x2 gx = f2_sub(one, cx.f), gy = f2_sub(one, cy.f), gz = f2_sub(one, cz.f);
        const f32x2 v00 = f2_fma(c100, cx.f, f2_mul(c000, gx));
        const f32x2 v10 = f2_fma(c110, cx.f, f2_mul(c010, gx));
        const f32x2 v01 = f2_fma(c101, cx.f, f2_mul(c001, gx));
        const f32x2 v11 = f2_fma(c111, cx.f, f2_mul(c011, gx));
        const f32x2 v0 = f2_fma(v10, cy.f, f2_mul(v00, gy));
        const f32x2 v1 = f2_fma(v11, cy.f, f2_mul(v01, gy));
        return f2_fma(v1, cz.f, f2_mul(v0, gz));
    }
};

// c = d / den, 0 where den is exactly 0 (the quotient of `term`)
__device__ __forceinline__ f32x2 pair_quotient(f32x2 d, f32x2 den) {
    float da, db, na, nb;
    f2_unpack(den, da, db);
    f2_unpack(d, na, nb);
    return f2_pack(da == 0.0f ? 0.0f : r_div(na, da), db == 0.0f ? 0.0f : r_div(nb, db));
}

// The update of Eqs. (1)-(6) at two voxels, demons_force<float, V> lane by
// lane: v = u - dr, and dr itself for the reductions.  Where dr is one term
// c * g, v is one fused multiply-add from c, which is how the scalar kernels'
// u - c * g is rounded; a sum of two terms is rounded before it is subtracted.
template <int V>
__device__ __forceinline__ void pair_update(f32x2 d, const f32x2 (&gs)[3], const f32x2 (&gm)[3],
                                            f32x2 b, float alpha2, const f32x2 (&u)[3],
                                            f32x2 (&dr)[3], f32x2 (&v)[3]) {
    // d^2 (Eq. 5: alpha^2 d^2) is rounded by itself before |g|^2 is added, as
    // the compiler contracts the scalar kernels, which use it twice
    if (V == 3 || V == 4) {
        f32x2 d2 = f2_mul(d, d);
        if (V == 4) d2 = f2_mul(f2_dup(alpha2), d2);
        const f32x2 p = pair_quotient(d, f2_add_rounded(d2, f2_sq3(gs[0], gs[1], gs[2])));
        const f32x2 q = pair_quotient(d, f2_add_rounded(d2, f2_sq3(gm[0], gm[1], gm[2])));
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            dr[c] = f2_add_rounded(f2_mul(p, gs[c]), f2_mul(q, gm[c]));
            v[c] = f2_sub_rounded(u[c], dr[c]);
        }
        return;
    }
    const f32x2(&g)[3] = (V == 2 || V == 5) ? gm : gs;
    f32x2 q;
    if (V == 1) {
        const f32x2 gs2 = f2_sq3(g[0], g[1], g[2]);
        float ga, gb;
        f2_unpack(gs2, ga, gb);
        const f32x2 a = f2_pack(r_sqrt(ga), r_sqrt(gb));
        const f32x2 s = f2_fma(b, b, f2_mul(a, a));
        const f32x2 den = f2_mul(f2_fma(f2_dup(2.0f), f2_mul(d, d), s), s);
        q = pair_quotient(f2_mul(f2_mul(f2_mul(f2_dup(4.0f), d), a), b), den);
    } else {
        q = pair_quotient(d, f2_add_rounded(f2_mul(d, d), f2_sq3(g[0], g[1], g[2])));
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        dr[c] = f2_mul(q, g[c]);
        v[c] = f2_sub_rounded(u[c], dr[c]);
    }
}

// The reductions of one thread: sum d^2, sum |du|, sum |u| over its voxels.  The
// norms are the scalar kernels' (r_norm_fast): not a number where the square
// overflows, so that no stop test takes it for convergence, and right for
// subnormal squares.
struct PairSums {
    float d2 = 0.0f, du = 0.0f, u = 0.0f;
    __device__ __forceinline__ void add(f32x2 d, const f32x2 (&dr)[3], const f32x2 (&uu)[3], bool va,
                                        bool vb) {
        float da, db, wa, wb, sa, sb;
        f2_unpack(d, da, db);
        f2_unpack(f2_sq3_yxz(dr[0], dr[1], dr[2]), wa, wb);
        f2_unpack(f2_sq3_yxz(uu[0], uu[1], uu[2]), sa, sb);
        if (va) {
            d2 = fmaf(da, da, d2);
            du += r_norm_fast(wa);
            u += r_norm_fast(sa);
        }
        if (vb) {
            d2 = fmaf(db, db, d2);
            du += r_norm_fast(wb);
            u += r_norm_fast(sb);
        }
    }
};

// The z pass of the Gaussian (radius R) down a column of t in shared memory,
// plane j at col[j * stride]: u at the FTZ middle planes, as pairs (k, k + H).
// Taps oldest plane first, fused multiply-adds from zero, as smooth2_kernel.
template <int R, int FTZ, int H>
__device__ __forceinline__ void pair_zpass(const float* col, int stride, const Taps& taps,
                                           f32x2 (&u)[H]) {
    constexpr int HB = FTZ > 1 ? H : 0;
    f32x2 c[H + 2 * R];
#pragma unroll
    for (int j = 0; j < H + 2 * R; ++j) c[j] = f2_pack(col[j * stride], col[(j + HB) * stride]);
#pragma unroll
    for (int k = 0; k < H; ++k) {
        u[k] = 0ull;
#pragma unroll
        for (int t = 0; t < 2 * R + 1; ++t) {
            const float2 w = taps.wp[t <= R ? t : 2 * R - t];
            u[k] = f2_fma(f2_pack(w.x, w.y), c[k + t], u[k]);
        }
    }
}

// A column of zero-filled box planes outside the volume, replicated from the
// nearest plane inside: planes jlo .. jhi of np are in the volume.  Only the
// thread that owns the column reads or writes it.
template <typename T>
__device__ __forceinline__ void replicate_planes(T* col, int stride, int np, int jlo, int jhi) {
    const T lo = col[jlo * stride], hi = col[jhi * stride];
    for (int j = 0; j < jlo; ++j) col[j * stride] = lo;
    for (int j = jhi + 1; j < np; ++j) col[j * stride] = hi;
}

}  // namespace dirk
