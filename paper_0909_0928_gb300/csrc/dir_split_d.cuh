// dir_split_d.cuh -- the Eqs. (3)-(6) iteration split once more, after the
// difference image: D = W - S is formed once per voxel instead of once per
// voxel of every block footprint that reaches it.
//
// The force of Eqs. 3-6 needs the gradient of the warped image, so a block of
// the one-pass form (dir_force_gm.cuh) interpolates W on its brick plus a
// one-voxel halo: about twice per voxel at 32 x 8 x 4 bricks, four times for
// Eq. 6, which also warps S backwards.  Here one iteration is three kernels:
//   x/y pass   t = G_y G_x v                     (dir_xy.cuh, sxy_block)
//   z + D pass u = G_z t down each thread's own column, then per voxel
//              D = W - S (Eq. 6: D_m + D_s and d = D_m - D_s); writes D
//   force pass u = G_z t again, the gradients of S and of W (= D + S) from
//              shared-memory boxes of D and S with a one-voxel halo, the
//              force, v = u - dr(u) and the reductions: a stencil with no
//              gathers
// The arithmetic is that of gm_force_body voxel by voxel (D by the same
// interpolation with the same operands, the same clamped neighbours, the same
// force), so the field is bit for bit the one of the other schedules.  The
// default for Eqs. 3-6 on every pyramid level: the one-pass blocks were bound by
// issue and by the latency of their footprint gathers, not by memory.
//
// With packed arithmetic (dir_pair.cuh) these kernels run at 0.86 of the copy
// rate on large levels, so u does not cross memory between them there: the
// force pass redoes the z pass (24 warp instructions per 32 voxels) instead of
// reading a u that the z + D pass would write, 80 B per voxel and iteration
// instead of 92 (Eq. 6: 88 for 100).  On levels that stay in L2 the second z
// pass only lengthens the chain, and the z + D pass writes u too (UW; the rule
// is force_d_writes_u).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "dir_force_kernel.cuh"
#include "dir_split.cuh"

namespace dirk {

// z + D pass: the brick of t with R planes above and below (as FZGeom).
template <int FTZ>
struct ZDGeom {
    static constexpr int NPZ = FTZ + 2 * FZR;
    static constexpr int TBOX = 3 * NPZ * FTY * FTX * 4;  // [3][NPZ][FTY][FTX] floats
    static constexpr int OFF_BAR = (TBOX + 127) / 128 * 128;
    static constexpr int SMEM = 128 + OFF_BAR + 64;
};

// One brick of the z + D pass (every thread of the block calls it).  a.u: t;
// a.dbuf: D out (Eq. 6: D_m + D_s), a.dbuf2: Eq. 6's d out; UW: a.v: u out.
template <int V, int FTZ, typename TI, bool UW>
__device__ __forceinline__ void zd_block(const CUtensorMap* tmap, const ForceArgs& a,
                                         const Taps& taps, const BlockPos bp) {
    static_assert(V >= 2 && V <= 5, "Eqs. 3-6");
    if (a.stop_iter != nullptr && *a.stop_iter < a.iter) return;  // uniform across the grid
    constexpr bool IC = (V == 5);
    using Z = ZDGeom<FTZ>;
    constexpr int R = FZR, NPZ = Z::NPZ;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    float* tb = reinterpret_cast<float*>(base);  // [3][NPZ][FTY][FTX]
    uint64_t* bar = reinterpret_cast<uint64_t*>(base + Z::OFF_BAR);
    const Grid3 g = a.g;
    const TI* __restrict__ S = static_cast<const TI*>(a.S);
    const TI* __restrict__ M = static_cast<const TI*>(a.M);
    float* __restrict__ uo = static_cast<float*>(a.v);
    float* __restrict__ Do = static_cast<float*>(a.dbuf);
    float* __restrict__ do2 = static_cast<float*>(a.dbuf2);
    const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + FTX * ty;
    // bricks from the top plane down, as zs_block (t was written bottom up)
    const int bx0 = bp.x * FTX, by0 = bp.y * FTY;
    const int bz0 = (bp.gz - 1 - bp.z) * FTZ;
    const int x = bx0 + tx, y = by0 + ty;
    const bool col_valid = (x < g.nx) && (y < g.ny);
    constexpr int H = FTZ > 1 ? FTZ / 2 : 1;  // pairs (k, k + H); FTZ = 1: both lanes the voxel
    constexpr int HB = FTZ > 1 ? H : 0;
    const uint32_t ipl = (uint32_t)sizeof(TI) * (uint32_t)g.plane;
    pdl_trigger();
    // S at this thread's voxels (static: read before the wait), planes past the
    // last as the last
    f32x2 s0[H];
#pragma unroll
    for (int k = 0; k < H; ++k) {
        const uint32_t o = (uint32_t)sizeof(TI) * (uint32_t)offs(g, min(x, g.nx - 1), min(y, g.ny - 1), 0);
        s0[k] = f2_pack(img_ldg(S, o + ipl * (uint32_t)min(bz0 + k, g.nz - 1)),
                        img_ldg(S, o + ipl * (uint32_t)min(bz0 + k + HB, g.nz - 1)));
    }
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
        fence_proxy_async();
        mbar_arrive_expect_tx(bar, (uint32_t)Z::TBOX);
        pdl_wait();
        tma_load_4d(base, tmap, bx0, by0, bz0 - R, 0, bar);  // planes outside: zero fill
        BlockPos nb;
        if (a.pf_stride > 0 && bp.ahead(a.pf_stride, nb))  // that block's t box into L2
            tma_prefetch_4d(tmap, nb.x * FTX, nb.y * FTY, (bp.gz - 1 - nb.z) * FTZ - R, 0);
    }
    pdl_wait();  // every thread: D is written below, which the previous iteration's
                 // force pass reads (finished before the kernel before)
    __syncthreads();
    // every thread waits for the copy itself (bounded); one that gave up flags
    // the error and goes on over whatever the box holds
    if (!mbar_wait_bounded(bar, 0, kWaitLimitNs) && a.err) atomicOr(a.err, kErrTmaTimeout);
    if (!col_valid) return;  // no barrier below

    // z pass down this thread's column, as zs_block
    float* tcol = tb + tid;  // plane j of component c at tcol[(c * NPZ + j) * FNT]
    const int zlo = bz0 - R;
    if (zlo < 0 || zlo + NPZ > g.nz)
        for (int c = 0; c < 3; ++c)
            replicate_planes(tcol + c * NPZ * FNT, FNT, NPZ, max(0, -zlo),
                             min(NPZ - 1, g.nz - 1 - zlo));
    f32x2 up[3][H];
#pragma unroll
    for (int c = 0; c < 3; ++c) pair_zpass<R, FTZ, H>(tcol + c * NPZ * FNT, FNT, taps, up[c]);

    // D per voxel: the interpolations of gm_force_body's d_at at the voxel itself
    const PairInterp<TI> ip(g, x, y, bz0);
    const uint32_t o0 = 4u * (uint32_t)offs(g, x, y, bz0), pl = 4u * (uint32_t)g.plane;
#pragma unroll
    for (int k = 0; k < H; ++k) {
        const int ka = k, kb = k + HB;
        const bool va = bz0 + ka < g.nz, vb = FTZ > 1 && bz0 + kb < g.nz;
        const f32x2 wm = ip.at(M, ka, kb, up[0][k], up[1][k], up[2][k], s0[k]);
        f32x2 D = wm, d = 0ull;
        if (IC) {
            const f32x2 ws =
                ip.at(S, ka, kb, f2_neg(up[0][k]), f2_neg(up[1][k]), f2_neg(up[2][k]), s0[k]);
            D = f2_add(wm, ws);
            d = f2_sub(wm, ws);
        }
        if (va) {
            const uint32_t o = o0 + ka * pl;
            if (UW) {
                *at_byte(uo, o) = f2_lo(up[0][k]);
                *at_byte(uo + g.cs, o) = f2_lo(up[1][k]);
                *at_byte(uo + 2 * g.cs, o) = f2_lo(up[2][k]);
            }
            *at_byte(Do, o) = f2_lo(D);
            if (IC) *at_byte(do2, o) = f2_lo(d);
        }
        if (vb) {
            const uint32_t o = o0 + kb * pl;
            if (UW) {
                *at_byte(uo, o) = f2_hi(up[0][k]);
                *at_byte(uo + g.cs, o) = f2_hi(up[1][k]);
                *at_byte(uo + 2 * g.cs, o) = f2_hi(up[2][k]);
            }
            *at_byte(Do, o) = f2_hi(D);
            if (IC) *at_byte(do2, o) = f2_hi(d);
        }
    }
}

// Force pass: D with a one-voxel halo over the columns x0 - 4 .. x0 + 35 (a
// 16-byte aligned start), S with the halo of FGGeom, t on the brick with R
// planes above and below (UW: u on the brick) and Eq. 6's d on the brick.
template <int FTZ, int V, typename TI, bool UW>
struct STGeom {
    static constexpr bool IC = (V == 5);
    static constexpr int FBX = 16 / (int)sizeof(TI);
    static constexpr int FSW = FTX + 2 * FBX;
    static constexpr int DW = FTX + 8, DH = FTY + 2, DD = FTZ + 2;
    static constexpr int DBOX = DD * DH * DW * 4;                    // [DD][DH][DW] floats
    static constexpr int SBOX = DD * FSH * FSW * (int)sizeof(TI);   // [DD][FSH][FSW]
    static constexpr int TR = UW ? 0 : FZR;                         // halo planes of t
    static constexpr int NPZ = FTZ + 2 * TR;
    static constexpr int TBOX = 3 * NPZ * FTY * FTX * 4;            // [3][NPZ][FTY][FTX]
    static constexpr int EBOX = IC ? FTZ * FTY * FTX * 4 : 0;       // [FTZ][FTY][FTX]
    static constexpr int OFF_S = (DBOX + 127) / 128 * 128;
    static constexpr int OFF_T = OFF_S + (SBOX + 127) / 128 * 128;
    static constexpr int OFF_E = OFF_T + (TBOX + 127) / 128 * 128;
    static constexpr int OFF_BAR = OFF_E + (EBOX + 127) / 128 * 128;
    static constexpr int SMEM = 128 + OFF_BAR + 64;
};

// One brick of the force pass (every thread of the block calls it).  a.u: t
// (UW: u), a.v: v out; a.dbuf: D, a.dbuf2: Eq. 6's d.
template <int V, int FTZ, typename TI, bool UW>
__device__ __forceinline__ void st_block(const CUtensorMap* dmap, const CUtensorMap* smap,
                                         const CUtensorMap* tmap, const CUtensorMap* emap,
                                         const ForceArgs& a, const Taps& taps, const BlockPos bp) {
    static_assert(V >= 2 && V <= 5, "Eqs. 3-6");
    if (a.stop_iter != nullptr && *a.stop_iter < a.iter) return;  // uniform across the grid
    using F = STGeom<FTZ, V, TI, UW>;
    constexpr int FSW = F::FSW, DW = F::DW, DH = F::DH, FBX = F::FBX;
    constexpr int R = F::TR, NPZ = F::NPZ;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    float* db = reinterpret_cast<float*>(base);                         // [DD][DH][DW]
    TI* sb = reinterpret_cast<TI*>(base + F::OFF_S);                    // [DD][FSH][FSW]
    float* tb = reinterpret_cast<float*>(base + F::OFF_T);              // [3][NPZ][FTY][FTX]
    const float* eb = reinterpret_cast<const float*>(base + F::OFF_E);  // [FTZ][FTY][FTX]
    uint64_t* bar = reinterpret_cast<uint64_t*>(base + F::OFF_BAR);
    const Grid3 g = a.g;
    float* __restrict__ v = static_cast<float*>(a.v);
    const float alpha2 = (float)a.alpha2;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = tx + FTX * ty;
    const int bx0 = bp.x * FTX, by0 = bp.y * FTY, bz0 = bp.z * FTZ;
    const int dx0 = bx0 - 4, dy0 = by0 - 1, dz0 = bz0 - 1;      // D box origin
    const int sx0 = bx0 - FBX, sy0 = by0 - 1, sz0 = bz0 - 1;    // S box origin
    pdl_trigger();
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
        fence_proxy_async();
        mbar_arrive_expect_tx(bar, (uint32_t)(F::DBOX + F::SBOX + F::TBOX + F::EBOX));
        tma_load_4d(base + F::OFF_S, smap, sx0, sy0, sz0, 0, bar);  // static
        pdl_wait();
        tma_load_4d(base, dmap, dx0, dy0, dz0, 0, bar);
        tma_load_4d(base + F::OFF_T, tmap, bx0, by0, bz0 - R, 0, bar);  // planes outside: zero fill
        if (F::IC) tma_load_4d(base + F::OFF_E, emap, bx0, by0, bz0, 0, bar);
        BlockPos nb;
        if (a.pf_stride > 0 && bp.ahead(a.pf_stride, nb)) {  // that block's boxes into L2
            const int px = nb.x * FTX, py = nb.y * FTY, pz = nb.z * FTZ;
            tma_prefetch_4d(dmap, px - 4, py - 1, pz - 1, 0);
            tma_prefetch_4d(smap, px - FBX, py - 1, pz - 1, 0);
            tma_prefetch_4d(tmap, px, py, pz - R, 0);
        }
    }
    pdl_wait();  // every thread: v is written below, which this iteration's x/y
                 // pass read (finished before the kernel before)
    __syncthreads();
    if (!mbar_wait_bounded(bar, 0, kWaitLimitNs) && a.err) atomicOr(a.err, kErrTmaTimeout);

    const int x = bx0 + tx, y = by0 + ty;
    PairSums sums;
    CorrSums<float> corr_s;  // with a.corr: the correlation sums
    if (x < g.nx && y < g.ny) {
        constexpr int SP = FSH * FSW, DP = DH * DW;  // elements per plane of the boxes
        constexpr int H = FTZ > 1 ? FTZ / 2 : 1, HB = FTZ > 1 ? H : 0;
        TI* scol = sb + (y - sy0) * FSW + (x - sx0);
        float* dcol = db + (y - dy0) * DW + (x - dx0);
        if (bz0 == 0 || bz0 + FTZ >= g.nz) {  // z neighbours outside the volume
            const int jlo = bz0 == 0 ? 1 : 0, jhi = min(FTZ + 1, g.nz - bz0);
            replicate_planes(scol, SP, FTZ + 2, jlo, jhi);
            replicate_planes(dcol, DP, FTZ + 2, jlo, jhi);
        }
        // x and y neighbours, clamped to the volume
        const int dxm = x > 0 ? -1 : 0, dxp = x < g.nx - 1 ? 1 : 0;
        const int yms = y > 0 ? -FSW : 0, yps = y < g.ny - 1 ? FSW : 0;
        const int ymd = y > 0 ? -DW : 0, ypd = y < g.ny - 1 ? DW : 0;
        float* __restrict__ vx = v;
        float* __restrict__ vy = v + g.cs;
        float* __restrict__ vz = v + 2 * g.cs;
        const uint32_t o0 = 4u * (uint32_t)offs(g, x, y, bz0), pl = 4u * (uint32_t)g.plane;
        const f32x2 half = f2_dup(0.5f), ns = f2_dup(F::IC ? 2.0f : 1.0f);
        // u down this thread's column, as zs_block
        float* tcol = tb + tid;
        f32x2 up[3][H];
        if constexpr (!UW) {
            if (bz0 < R || bz0 + FTZ + R > g.nz)
                for (int c = 0; c < 3; ++c)
                    replicate_planes(tcol + c * NPZ * FNT, FNT, NPZ, max(0, R - bz0),
                                     min(NPZ - 1, g.nz - 1 - bz0 + R));
#pragma unroll
            for (int c = 0; c < 3; ++c)
                pair_zpass<R, FTZ, H>(tcol + c * NPZ * FNT, FNT, taps, up[c]);
        }
        auto pairs = [&](auto whole) {  // whole: every plane of the brick lies in the volume
#pragma unroll
            for (int k = 0; k < H; ++k) {
                const int ka = k, kb = k + HB;
                const bool va = whole || bz0 + ka < g.nz;
                const bool vb = FTZ > 1 && (whole || bz0 + kb < g.nz);
                auto sgrad = [&](int dp, int dm) {  // half the difference of two values of S
                    const TI* pa = scol + (ka + 1) * SP;
                    const TI* pb = scol + (kb + 1) * SP;
                    return f2_mul(half, f2_sub(f2_pack(img_bits(pa[dp]), img_bits(pb[dp])),
                                               f2_pack(img_bits(pa[dm]), img_bits(pb[dm]))));
                };
                auto dgrad = [&](int dp, int dm) {  // and of D
                    const float* pa = dcol + (ka + 1) * DP;
                    const float* pb = dcol + (kb + 1) * DP;
                    return f2_mul(half, f2_sub(f2_pack(pa[dp], pb[dp]), f2_pack(pa[dm], pb[dm])));
                };
                const f32x2 gs[3] = {sgrad(dxp, dxm), sgrad(yps, yms), sgrad(SP, -SP)};
                // grad W = grad D + grad S (Eq. 6: grad(D_m + D_s) + 2 grad S)
                const f32x2 gm[3] = {f2_fma(ns, gs[0], dgrad(dxp, dxm)),
                                     f2_fma(ns, gs[1], dgrad(ypd, ymd)),
                                     f2_fma(ns, gs[2], dgrad(DP, -DP))};
                const f32x2 D = f2_pack(dcol[(ka + 1) * DP], dcol[(kb + 1) * DP]);
                const f32x2 d =
                    F::IC ? f2_pack(eb[tid + ka * FNT], eb[tid + kb * FNT]) : D;
                if (a.corr) {  // reference: S (Eq. 6: the warped static image S + D_s)
                    float ra = img_value<TI>(img_bits(scol[(ka + 1) * SP]));
                    float rb = img_value<TI>(img_bits(scol[(kb + 1) * SP]));
                    if (F::IC) {
                        ra += 0.5f * (f2_lo(D) - f2_lo(d));
                        rb += 0.5f * (f2_hi(D) - f2_hi(d));
                    }
                    if (va) corr_s.add(ra, f2_lo(d));
                    if (vb) corr_s.add(rb, f2_hi(d));
                }
                f32x2 u[3];
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    u[c] = UW ? f2_pack(tcol[(c * NPZ + ka) * FNT], tcol[(c * NPZ + kb) * FNT])
                              : up[c][k];
                f32x2 dr[3], vn[3];
                pair_update<V>(d, gs, gm, 0ull, alpha2, u, dr, vn);
                sums.add(d, dr, u, va, vb);
                if (va) {
                    const uint32_t o = o0 + ka * pl;
                    *at_byte(vx, o) = f2_lo(vn[0]);
                    *at_byte(vy, o) = f2_lo(vn[1]);
                    *at_byte(vz, o) = f2_lo(vn[2]);
                }
                if (vb) {
                    const uint32_t o = o0 + kb * pl;
                    *at_byte(vx, o) = f2_hi(vn[0]);
                    *at_byte(vy, o) = f2_hi(vn[1]);
                    *at_byte(vz, o) = f2_hi(vn[2]);
                }
            }
        };
        if (bz0 + FTZ <= g.nz)
            pairs(std::true_type{});
        else
            pairs(std::false_type{});
    }
    block_reduce3_atomic<FNT, float>(sums.d2, sums.du, sums.u, a.red);
    if (a.corr) block_reduce4_atomic<FNT, float>(corr_s, a.corr);
}

}  // namespace dirk
