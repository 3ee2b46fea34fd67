// dir_level.cu -- all iterations of a small pyramid level in one launch: a
// thread-block cluster keeps the level's field in its shared memory from the
// starting field to the level's result.
//
// A small level's iteration (two or three kernels of the split schedule) is a
// chain of latencies: launch, block start, copy from L2, passes, write, drain.
// 16x16x8 voxels take as long as 32x32x16 (4.9 us per passive iteration).  Here
// each CTA of the cluster owns a tile of TR rows x TP planes (all columns) and
// one iteration is
//   x pass  of v on the tile's rows and 3 halo rows each side    (own memory)
//   y pass  -> t on the tile, each value also stored into the halo planes of
//           the tiles above and below that will read it          (DSMEM stores)
//   cluster barrier
//   z pass  u = G_z t down the column, interpolation, force, v = u - dr(u),
//           each value also stored into the halo rows of the tiles beside it
//   cluster barrier
// with one barrier more for Eqs. (3)-(6), whose force differences D = W - S
// across tiles.  Halos are pushed by the CTA that makes them (stores that nobody
// waits for until the barrier), so every read is of the CTA's own memory; M (and
// S for Eq. 6's backward warp) is gathered through L1.  The arithmetic is that of
// the split kernels (dir_pair.cuh), voxel by voxel, so the field is bit for bit
// theirs.  Only the level's starting and resulting field touch global memory.
//
// Measured per iteration, split kernels -> this, Eq. 1 / Eq. 3: 16x16x8 4.84 ->
// 2.52 us / 6.5 -> 3.5, 25x25x10 4.9 -> 3.4 / 6.4 -> 4.4, 32x32x16 4.88 -> 3.92 /
// 6.35 -> 5.1; 48x43x22 (45,000 voxels) is faster split, so levels above 16,384
// voxels stay there.  What bounds it: a cluster barrier takes 0.5 us with the halo
// stores before it (two per iteration, three for Eqs. 3-6), the rest is one
// dependent chain per pass on a few warps per SM; at 32x32x16 the force itself
// (1.3 us) is issue bound.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "dir_launch.h"
#include "dir_once.h"
#include "dir_pair.cuh"
#include "dir_stencil.cuh"

namespace dirk {

namespace {

constexpr int LNT = 512;  // threads per CTA
constexpr int LR = 3;     // Gaussian radius
// Entries per plane (row) of the halo tables, a count and cluster addresses: a
// plane of t goes to its own tile, to the tiles within R planes, and, being the
// first or last of the volume, to the planes beyond it in those tiles
constexpr int kTz = 12, kVy = 8;

// Shared-memory layout of one CTA, in floats from the base (the same in every
// CTA of the cluster: halo stores use the receiver's offsets)
struct LevelGeom {
    int nx, nx4;           // columns, rounded up to 4
    int TR, TP;            // rows and planes of a tile
    int ncy, ncz;          // tiles along y and z
    int vp;                // v row pitch: 4 floats before the row and after it
    int sx;                // S and D row pitch: nx + 2
    int off_v, off_f, off_t, off_s, off_b, off_d, off_e, off_p, off_tz, off_vy;
    int floats;
    __host__ __device__ LevelGeom(const Grid3& g, int variant, int tr, int tp) {
        nx = g.nx;
        nx4 = (g.nx + 3) / 4 * 4;
        TR = tr;
        TP = tp;
        ncy = (g.ny + tr - 1) / tr;
        ncz = (g.nz + tp - 1) / tp;
        vp = nx4 + 8;
        sx = nx + 2;
        int o = 0;
        auto take = [&](int n) {
            const int at = o;
            o += (n + 3) / 4 * 4;
            return at;
        };
        off_v = take(3 * tp * (tr + 2 * LR) * vp);            // v: [3][TP][TR+6][vp]
        off_f = take(3 * tp * (tr + 2 * LR) * nx4);           // x-filtered rows; later u
        off_t = take(3 * (tp + 2 * LR) * tr * nx4);           // t: [3][TP+6][TR][nx4]
        off_s = take((tp + 2) * (tr + 2) * sx);               // S: [TP+2][TR+2][sx]
        off_b = variant == 1 ? take(tp * tr * nx) : o;        // |grad M|: [TP][TR][nx]
        off_d = variant >= 2 ? take((tp + 2) * (tr + 2) * sx) : o;  // D: as S
        off_e = variant == 5 ? take(tp * tr * nx) : o;        // Eq. 6's d: [TP][TR][nx]
        off_p = take(3 * LNT);                                // per-thread sums of an iteration
        off_tz = take(tp * kTz);                              // where the planes of t go
        off_vy = take(tr * kVy);                              // where the rows of v go, besides here
        floats = o;
    }
};

__device__ __forceinline__ uint32_t cluster_addr(uint32_t own, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(own), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_store(uint32_t addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_store(uint32_t addr, float4 v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x),
                 "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}
// All threads of all CTAs of the cluster; what each stored before (its own and
// other CTAs' shared memory) is visible to all after.
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

template <int V, typename TI>
__global__ void __launch_bounds__(LNT, 1) level_kernel(const __grid_constant__ LevelGroup G) {
    constexpr bool GM = V >= 2, IC = V == 5;
    constexpr int R = LR, K = 2 * R + 1;
    extern __shared__ float4 smem4[];
    float* const sm = reinterpret_cast<float*>(smem4);
    const uint32_t sm_addr = smem_u32(sm);
    const int job = blockIdx.x / G.cluster;
    const int rank = blockIdx.x - job * G.cluster;  // rank in the cluster
    const LevelArgs& a = G.a[job];
    const Taps& taps = G.taps;
    const Grid3 g = a.g;
    const LevelGeom L(g, V, a.tile_rows, a.tile_planes);
    const int TR = L.TR, TP = L.TP, nx = L.nx, nx4 = L.nx4;
    const int cy = rank % L.ncy, cz = rank / L.ncy;  // cz >= ncz: a CTA without voxels
    const int y0 = cy * TR, z0 = cz * TP;
    const int rows = cz < L.ncz ? min(TR, g.ny - y0) : 0;
    const int planes = cz < L.ncz ? min(TP, g.nz - z0) : 0;
    const int tid = threadIdx.x;
    const TI* __restrict__ S = static_cast<const TI*>(a.S);
    const TI* __restrict__ M = static_cast<const TI*>(a.M);

    // S on the tile and one voxel around it, clamped (img_bits form); Eq. 2: |grad M|
    const int ns = rows > 0 ? (planes + 2) * (rows + 2) * L.sx : 0;
    for (int i = tid; i < ns; i += LNT) {
        const int x = i % L.sx, q = i / L.sx, r = q % (rows + 2), p = q / (rows + 2);
        const int o = offs(g, clampi(x - 1, 0, nx - 1), clampi(y0 + r - 1, 0, g.ny - 1),
                           clampi(z0 + p - 1, 0, g.nz - 1));
        sm[L.off_s + (p * (TR + 2) + r) * L.sx + x] = img_bits(__ldg(S + o));
    }
    if (V == 1) {
        for (int i = tid; i < nx * rows * planes; i += LNT) {
            const int x = i % nx, q = i / nx, y = y0 + q % rows, z = z0 + q / rows;
            auto at = [&](int X, int Y, int Z) { return img_bits(__ldg(M + offs(g, X, Y, Z))); };
            const float mx = 0.5f * (at(min(x + 1, nx - 1), y, z) - at(max(x - 1, 0), y, z));
            const float my = 0.5f * (at(x, min(y + 1, g.ny - 1), z) - at(x, max(y - 1, 0), z));
            const float mz = 0.5f * (at(x, y, min(z + 1, g.nz - 1)) - at(x, y, max(z - 1, 0)));
            sm[L.off_b + ((z - z0) * TR + (y - y0)) * nx + x] =
                f2_lo(f2_norm_yxz(f2_dup(mx), f2_dup(my), f2_dup(mz)));
        }
    }
    // halo tables (cluster addresses of the first column, of component 0; t: row 0)
    uint32_t* const tz = reinterpret_cast<uint32_t*>(sm + L.off_tz);
    uint32_t* const vy = reinterpret_cast<uint32_t*>(sm + L.off_vy);
    for (int pl = tid; pl < planes; pl += LNT) {
        const int z = z0 + pl, zb = z == 0 ? -R : z, ze = z == g.nz - 1 ? z + R : z;
        uint32_t n = 0;
        for (int gz = zb; gz <= ze; ++gz) {
            const int lo = gz >= R ? (gz - R) / TP : 0, hi = min((gz + R) / TP, L.ncz - 1);
            for (int cc = lo; cc <= hi; ++cc)
                tz[pl * kTz + 1 + n++] = cluster_addr(
                    sm_addr + 4u * (L.off_t + (gz - cc * TP + R) * TR * nx4), cy + L.ncy * cc);
        }
        tz[pl * kTz] = n;
    }
    for (int r = tid; r < rows; r += LNT) {
        const int y = y0 + r, lo = y >= R ? (y - R) / TR : 0, hi = min((y + R) / TR, L.ncy - 1);
        uint32_t n = 0;
        for (int cc = lo; cc <= hi; ++cc)
            if (cc != cy)
                vy[r * kVy + 1 + n++] = cluster_addr(
                    sm_addr + 4u * (L.off_v + (y - cc * TR + R) * L.vp + 4), cc + L.ncy * cz);
        vy[r * kVy] = n;
    }

    // A thread's tasks in each loop: the digits of its first one, found once, and
    // of the step to its next (LNT further on), so that no loop divides.  Digits
    // of an all-zero radix belong to a CTA without voxels, whose loops are empty.
    const int g4 = nx4 / 4;
    const int lr0 = max(0, R - y0), lr1 = min(rows + 2 * R, g.ny - y0 + R);  // rows in the volume
    const int H = (planes + 1) / 2;  // items: voxel pairs, planes p and p + H of one column
    struct Digits {
        int a, b, c;
        __device__ Digits(int i, int na, int nb) {
            const int q = i / max(na, 1);
            a = i - q * na;
            c = q / max(nb, 1);
            b = q - c * nb;
        }
        __device__ void step(const Digits& d, int na, int nb) {
            a += d.a;
            b += d.b;
            c += d.c;
            if (a >= na) {
                a -= na;
                b += 1;
            }
            if (b >= nb) {
                b -= nb;
                c += 1;
            }
        }
    };
    const Digits x_first(tid, g4, lr1 - lr0), x_step(LNT, g4, lr1 - lr0);
    const Digits y_first(tid, g4, rows), y_step(LNT, g4, rows);
    const Digits i_first(tid, nx, rows), i_step(LNT, nx, rows);
    cluster_barrier();  // every CTA runs: its shared memory may be written

    // x pass of v on the tile's rows and halo rows
    auto smooth_x = [&]() {
        Digits q = x_first;
        for (; q.c < 3 * planes; q.step(x_step, g4, lr1 - lr0)) {
            const int gx = q.a, lr = lr0 + q.b;
            const float4* v4 = reinterpret_cast<const float4*>(
                sm + L.off_v + (q.c * (TR + 2 * R) + lr) * L.vp + 4 * gx);
            const float4 p = v4[0], c = v4[1], n = v4[2];
            float in[12] = {p.x, p.y, p.z, p.w, c.x, c.y, c.z, c.w, n.x, n.y, n.z, n.w};
            if (gx == 0) in[1] = in[2] = in[3] = in[4];
            const int last = nx - 1 - 4 * gx;  // the volume's last column among in[4 + ..]
            if (last < 6) {
#pragma unroll
                for (int j = 1; j < 7; ++j) in[4 + j] = j > last ? in[3 + j] : in[4 + j];
            }
            float f[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                f[j] = 0.0f;
#pragma unroll
                for (int t = 0; t < K; ++t)
                    f[j] = fmaf(taps.wf[t <= R ? t : 2 * R - t], in[4 - R + j + t], f[j]);
            }
            const float4 out = make_float4(f[0], f[1], f[2], f[3]);
            float4* f4 = reinterpret_cast<float4*>(sm + L.off_f + q.c * (TR + 2 * R) * nx4) + gx;
            f4[lr * g4] = out;
            if (lr == lr0)  // rows before the first and past the last: the nearest row's
                for (int k = 0; k < lr0; ++k) f4[k * g4] = out;
            if (lr == lr1 - 1)
                for (int k = lr1; k < rows + 2 * R; ++k) f4[k * g4] = out;
        }
    };
    // y pass; t into this tile and the halo planes of others
    auto smooth_y = [&]() {
        Digits w = y_first;
        for (; w.c < 3 * planes; w.step(y_step, g4, rows)) {
            const int gx = w.a, r = w.b;
            const int c = w.c >= 2 * planes ? 2 : (w.c >= planes ? 1 : 0), pl = w.c - c * planes;
            const float4* f4 = reinterpret_cast<const float4*>(
                sm + L.off_f + (w.c * (TR + 2 * R) + r) * nx4) + gx;
            f32x2 v0 = 0ull, v1 = 0ull;
#pragma unroll
            for (int t = 0; t < K; ++t) {
                const float4 in = f4[t * g4];
                const float2 w2 = taps.wp[t <= R ? t : 2 * R - t];
                const f32x2 wt = f2_pack(w2.x, w2.y);
                v0 = f2_fma(wt, f2_pack(in.x, in.y), v0);
                v1 = f2_fma(wt, f2_pack(in.z, in.w), v1);
            }
            const float4 out = make_float4(f2_lo(v0), f2_hi(v0), f2_lo(v1), f2_hi(v1));
            const uint32_t at = 4u * ((c * (TP + 2 * R) * TR + r) * nx4 + 4 * gx);
            const uint32_t* to = tz + pl * kTz;
            const int n = (int)to[0];
            for (int k = 1; k <= n; ++k) cluster_store(to[k] + at, out);
        }
    };

    // v of one voxel (lane) into this tile and the halo rows of the tiles beside it
    auto put_v = [&](int x, int r, int pl, float vx, float vy_, float vz) {
        const int step = planes * (TR + 2 * R) * L.vp;  // floats per component
        const int col = pl * (TR + 2 * R) * L.vp + x;
        float* v = sm + L.off_v + (r + R) * L.vp + 4 + col;
        v[0] = vx;
        v[step] = vy_;
        v[2 * step] = vz;
        const uint32_t* to = vy + r * kVy;
        const int n = (int)to[0];
        for (int k = 1; k <= n; ++k) {
            const uint32_t ad = to[k] + 4u * col;
            cluster_store(ad, vx);
            cluster_store(ad + 4u * step, vy_);
            cluster_store(ad + 8u * step, vz);
        }
    };
    // D of one voxel into this tile and the halo cells that hold it
    auto put_d = [&](int x, int r, int pl, float d) {
        const int row = L.sx, pln = (TR + 2) * L.sx;
        const int at = L.off_d + ((pl + 1) * (TR + 2) + r + 1) * L.sx + x + 1;
        const int y = y0 + r, z = z0 + pl;
        sm[at] = d;
        if (x == 0) sm[at - 1] = d;
        if (x == nx - 1) sm[at + 1] = d;
        auto send = [&](int to, int tile_y, int tile_z) {
            cluster_store(cluster_addr(sm_addr + 4u * to, tile_y + L.ncy * tile_z), d);
        };
        // the tile before this one along an axis is always a whole one
        if (y == 0)
            sm[at - row] = d;
        else if (r == 0)
            send(at + TR * row, cy - 1, cz);
        if (y == g.ny - 1)
            sm[at + row] = d;
        else if (r == rows - 1)
            send(at - TR * row, cy + 1, cz);
        if (z == 0)
            sm[at - pln] = d;
        else if (pl == 0)
            send(at + TP * pln, cy, cz - 1);
        if (z == g.nz - 1)
            sm[at + pln] = d;
        else if (pl == planes - 1)
            send(at - TP * pln, cy, cz + 1);
    };

    const f32x2 half = f2_dup(0.5f);
    const int SP = (TR + 2) * L.sx;  // floats per plane of S and D
    auto u_of = [&](int x, int r, int pa, int pb, bool from_global, f32x2(&u)[3]) {
        if (from_global) {
            const float* up = a.u;
            const int oa = offs(g, x, y0 + r, z0 + pa), ob = offs(g, x, y0 + r, z0 + pb);
#pragma unroll
            for (int c = 0; c < 3; ++c) u[c] = f2_pack(up[c * g.cs + oa], up[c * g.cs + ob]);
            return;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float* ta = sm + L.off_t + ((c * (TP + 2 * R) + pa) * TR + r) * nx4 + x;
            const int db = (pb - pa) * TR * nx4;
            u[c] = 0ull;
#pragma unroll
            for (int t = 0; t < K; ++t) {
                const float2 w = taps.wp[t <= R ? t : 2 * R - t];
                u[c] = f2_fma(f2_pack(w.x, w.y), f2_pack(ta[t * TR * nx4], ta[t * TR * nx4 + db]),
                              u[c]);
            }
        }
    };
    auto grad3 = [&](const float* ca, const float* cb, f32x2(&o)[3]) {
        const int d[3] = {1, L.sx, SP};
#pragma unroll
        for (int c = 0; c < 3; ++c)
            o[c] = f2_mul(half, f2_sub(f2_pack(ca[d[c]], cb[d[c]]), f2_pack(ca[-d[c]], cb[-d[c]])));
    };

    // The sums of an iteration: every thread leaves its own in shared memory, and
    // the last three warps, which have the fewest tasks, add up one sum each during
    // the x pass (a lane those of 16 threads) and the y pass (over the lanes) of the
    // next iteration, FP64 across CTAs.  What an addition rounds away is kept beside
    // the sum (Knuth's TwoSum; FP64 runs at 1/64 of the rate): beyond a thread
    // nothing is lost to FP32, whose plain additions over 64 threads doubled the
    // error of the sums (sum d^2 at 32x32x16 against 64 bits: 3.5e-9, 1.8e-9 in the
    // split kernels, now 1.1e-9).
    float* const part = sm + L.off_p;
    const int lane = tid & 31, sum_of = (tid >> 5) - (LNT / 32 - 3);  // 0 .. 2, else negative
    float sum_hi = 0.0f, sum_lo = 0.0f;
    auto add = [&](float v) {
        const float t = __fadd_rn(sum_hi, v), b = __fsub_rn(t, sum_hi);
        sum_lo += __fadd_rn(__fsub_rn(sum_hi, __fsub_rn(t, b)), __fsub_rn(v, b));
        sum_hi = t;
    };
    auto reduce_threads = [&]() {
        if (sum_of < 0) return;
        const float4* p = reinterpret_cast<const float4*>(part + sum_of * LNT) + lane;
        sum_hi = sum_lo = 0.0f;
#pragma unroll
        for (int q = 0; q < LNT / 128; ++q) {
            const float4 v = p[32 * q];
            add(v.x);
            add(v.y);
            add(v.z);
            add(v.w);
        }
    };
    auto reduce_lanes = [&](int it) {
        if (sum_of < 0) return;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float hi = __shfl_down_sync(0xffffffffu, sum_hi, o);
            const float lo = __shfl_down_sync(0xffffffffu, sum_lo, o);
            add(hi);
            sum_lo += lo;
        }
        // an infinite sum leaves infinity - infinity in what was rounded away
        if (lane == 0)
            atomicAdd(a.red + 3 * it + sum_of,
                      isfinite(sum_hi) ? (double)sum_hi + (double)sum_lo : (double)sum_hi);
    };

    for (int it = 0; it < a.iters; ++it) {
        if (it > 0) {
            reduce_threads();
            smooth_x();
            __syncthreads();
            reduce_lanes(it - 1);
            smooth_y();
            cluster_barrier();
        }
        PairSums sums;
        CorrSums<float> corr_s;
        // the force and update of one pair, its D and S in shared memory
        auto update = [&](int x, int r, int pa, int pb, bool vb, f32x2 d, f32x2 ref,
                          const f32x2(&gm)[3], const f32x2(&gs)[3], const f32x2(&u)[3]) {
            f32x2 b = 0ull, dr[3], v[3];
            if (V == 1)
                b = f2_pack(sm[L.off_b + (pa * TR + r) * nx + x], sm[L.off_b + (pb * TR + r) * nx + x]);
            if (a.corr) {
                corr_s.add(f2_lo(ref), f2_lo(d));
                if (vb) corr_s.add(f2_hi(ref), f2_hi(d));
            }
            pair_update<V>(d, gs, gm, b, a.alpha2, u, dr, v);
            sums.add(d, dr, u, true, vb);
            put_v(x, r, pa, f2_lo(v[0]), f2_lo(v[1]), f2_lo(v[2]));
            if (vb) put_v(x, r, pb, f2_hi(v[0]), f2_hi(v[1]), f2_hi(v[2]));
        };
        for (Digits q = i_first; q.c < H; q.step(i_step, nx, rows)) {
            const int x = q.a, r = q.b, pa = q.c;
            const bool vb = pa + H < planes;
            const int pb = vb ? pa + H : pa;
            f32x2 u[3];
            u_of(x, r, pa, pb, it == 0, u);
            const float* sa = sm + L.off_s + ((pa + 1) * (TR + 2) + r + 1) * L.sx + x + 1;
            const float* sb = sa + (pb - pa) * SP;
            const f32x2 s0 = f2_pack(*sa, *sb);
            const PairInterp<TI> ip(g, x, y0 + r, z0);
            const f32x2 wm = ip.at(M, pa, pb, u[0], u[1], u[2], s0);
            if (!GM) {
                f32x2 gs[3];
                grad3(sa, sb, gs);
                update(x, r, pa, pb, vb, wm,
                       f2_pack(img_value<TI>(f2_lo(s0)), img_value<TI>(f2_hi(s0))), gs, gs, u);
            } else {
                f32x2 D = wm;
                if (IC) {
                    const f32x2 ws = ip.at(S, pa, pb, f2_neg(u[0]), f2_neg(u[1]), f2_neg(u[2]), s0);
                    D = f2_add(wm, ws);
                    const f32x2 e = f2_sub(wm, ws);
                    sm[L.off_e + (pa * TR + r) * nx + x] = f2_lo(e);
                    sm[L.off_e + (pb * TR + r) * nx + x] = vb ? f2_hi(e) : f2_lo(e);
                }
                put_d(x, r, pa, f2_lo(D));
                if (vb) put_d(x, r, pb, f2_hi(D));
                // u waits for the force where the x-filtered rows were
                float* ua = sm + L.off_f + (pa * TR + r) * nx4 + x;
                float* ub = sm + L.off_f + (pb * TR + r) * nx4 + x;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    ua[c * TP * TR * nx4] = f2_lo(u[c]);
                    if (vb) ub[c * TP * TR * nx4] = f2_hi(u[c]);
                }
            }
        }
        if (GM) {
            cluster_barrier();
            for (Digits q = i_first; q.c < H; q.step(i_step, nx, rows)) {
                const int x = q.a, r = q.b, pa = q.c;
                const bool vb = pa + H < planes;
                const int pb = vb ? pa + H : pa;
                const int ca = ((pa + 1) * (TR + 2) + r + 1) * L.sx + x + 1;
                const int cb = ca + (pb - pa) * SP;
                f32x2 gs[3], gd[3], gm[3], u[3];
                grad3(sm + L.off_s + ca, sm + L.off_s + cb, gs);
                grad3(sm + L.off_d + ca, sm + L.off_d + cb, gd);
                const f32x2 ns2 = f2_dup(IC ? 2.0f : 1.0f);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    gm[c] = f2_fma(ns2, gs[c], gd[c]);
                    const float* up = sm + L.off_f + ((c * TP + pa) * TR + r) * nx4 + x;
                    u[c] = f2_pack(up[0], up[(pb - pa) * TR * nx4]);
                }
                const f32x2 D = f2_pack(sm[L.off_d + ca], sm[L.off_d + cb]);
                f32x2 d = D;
                float ra = img_value<TI>(sm[L.off_s + ca]), rb = img_value<TI>(sm[L.off_s + cb]);
                if (IC) {
                    d = f2_pack(sm[L.off_e + (pa * TR + r) * nx + x],
                                sm[L.off_e + (pb * TR + r) * nx + x]);
                    ra += 0.5f * (f2_lo(D) - f2_lo(d));
                    rb += 0.5f * (f2_hi(D) - f2_hi(d));
                }
                update(x, r, pa, pb, vb, d, f2_pack(ra, rb), gm, gs, u);
            }
        }
        part[tid] = sums.d2;
        part[LNT + tid] = sums.du;
        part[2 * LNT + tid] = sums.u;
        if (a.corr) block_reduce4_atomic<LNT, float, 8>(corr_s, a.corr + 4 * it);
        cluster_barrier();
    }
    // the level's result: u = G v of the last iteration
    reduce_threads();
    smooth_x();
    __syncthreads();
    reduce_lanes(a.iters - 1);
    smooth_y();
    cluster_barrier();
    for (Digits q = i_first; q.c < H; q.step(i_step, nx, rows)) {
        const int x = q.a, r = q.b, pa = q.c;
        const bool vb = pa + H < planes;
        const int pb = vb ? pa + H : pa;
        f32x2 u[3];
        u_of(x, r, pa, pb, false, u);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            a.u[c * g.cs + offs(g, x, y0 + r, z0 + pa)] = f2_lo(u[c]);
            if (vb) a.u[c * g.cs + offs(g, x, y0 + r, z0 + pb)] = f2_hi(u[c]);
        }
    }
}

constexpr int kLevelMaxSmem = 220 * 1024;

// Tiles of a level for a cluster of C CTAs: the split over y and z with the least
// work on the largest tile (counted in warp instructions), of those that fit.
bool level_tiles(const Grid3& g, int variant, int C, int* tr, int* tp, int* smem) {
    double best = 1e30;
    for (int cy = 1; cy <= C; ++cy) {
        if (cy > g.ny) break;
        const int cz = std::min(C / cy, g.nz);
        const int TR = (g.ny + cy - 1) / cy, TP = (g.nz + cz - 1) / cz;
        const LevelGeom L(g, variant, TR, TP);
        if (L.ncy * L.ncz > C || (size_t)L.floats * 4 > (size_t)kLevelMaxSmem) continue;
        // per group of 4 columns: x and y pass, and a 16-byte store to each tile that
        // holds the plane as a halo; per voxel: the force, and 4-byte halo stores
        // (other CTAs' memory takes about 32 bytes per cycle)
        const double t4 = 3.0 * TP * TR * (L.nx4 / 4), col = (double)L.nx * TR * TP;
        const double work = 60.0 * t4 * (TR + 2 * LR) / TR + t4 * (40.0 + 60.0 * 2 * LR / TP) +
                            col * (170.0 + 45.0 * 2 * LR / TR);
        if (work < best) {
            best = work;
            *tr = TR;
            *tp = TP;
            *smem = L.floats * 4;
        }
    }
    return best < 1e30;
}

template <int V, typename TI>
cudaError_t setup_level() {
    static KernelSetup setup;  // per instantiation
    const cudaError_t e = setup_kernel(setup, level_kernel<V, TI>, kLevelMaxSmem);
    return e != cudaSuccess ? e
                            : cudaFuncSetAttribute(
                                  level_kernel<V, TI>,
                                  cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

// How many clusters of 1 .. kLevelCluster CTAs the current device runs at once
// (one CTA per SM; a cluster stays within a GPC), asked once per device; nullptr
// where it holds none of kLevelCluster / 2 CTAs (e.g. a partitioned GPU).
struct ActiveClusters {
    int n[kLevelCluster + 1];
};
const ActiveClusters* active_clusters() {
    static OncePerDevice<ActiveClusters, KernelSetup::kMaxDevices> table;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    const ActiveClusters* t = table.get(dev, [](ActiveClusters& t) {
        const bool ok = setup_level<0, float>() == cudaSuccess;
        for (int C = 1; C <= kLevelCluster; ++C) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = (unsigned)C;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            cfg.gridDim = dim3((unsigned)C);
            cfg.blockDim = dim3(LNT);
            cfg.dynamicSmemBytes = kLevelMaxSmem;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int n = 0;
            if (!ok ||
                cudaOccupancyMaxActiveClusters(&n, level_kernel<0, float>, &cfg) != cudaSuccess)
                n = 0;
            t.n[C] = n;
        }
        cudaGetLastError();
    });
    return t && t->n[kLevelCluster / 2] > 0 ? t : nullptr;
}

template <int V, typename TI>
cudaError_t launch_level_v(const LevelGroup& G, int smem, cudaStream_t s) {
    const cudaError_t e = setup_level<V, TI>();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(G.n * G.cluster));
    cfg.blockDim = dim3(LNT);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)G.cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, level_kernel<V, TI>, G);
}

template <typename TI>
cudaError_t launch_level_types(int variant, const LevelGroup& G, int smem, cudaStream_t s) {
    switch (variant) {
        case 0: return launch_level_v<0, TI>(G, smem, s);
        case 1: return launch_level_v<1, TI>(G, smem, s);
        case 2: return launch_level_v<2, TI>(G, smem, s);
        case 3: return launch_level_v<3, TI>(G, smem, s);
        case 4: return launch_level_v<4, TI>(G, smem, s);
        case 5: return launch_level_v<5, TI>(G, smem, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// CTAs per cluster for a launch over n levels.  An iteration takes about 1.6 us +
// 0.04 us per CTA (barriers) + 0.002 us per voxel of the largest tile (Eq. 1,
// measured / this: 16x16x8 16 CTAs 2.66 / 2.5, 8: 2.48 / 2.4, 6: 2.76 / 2.7, 5: 3.0;
// 32x32x16 16: 3.83 / 4.3, 8: 5.9 / 6.0, 6: 7.7 / 7.3), and clusters that do not
// run at once take turns.  A GB300 holds 7 clusters of 16 CTAs, 15 of 8, 23 of 6:
// 16 levels of 32x32x16 took 11.8 us an iteration in two turns of 8 CTAs and
// take 7.9 in one of 6 (the grouped split kernels: 10.4); 8 levels of 16x16x8
// 5.3 us in two turns of 16, now 2.5 in one of 8.  The same model serves the laws
// with a third barrier: its choice is the fastest of 4 to 16 CTAs, or within 2 %
// of it, for Eqs. 3 and 6 too (16x16x8 alone 8: 3.48 / 3.72 us, 16: 3.47 / 3.72;
// 32x32x16 alone 16: 5.1 / 5.7, 12: 6.8 / 7.3; 16 of 25x25x10 6: 7.0 / 7.8, 12: 10.1
// / 11.1; 16 of 32x32x16 6: 10.1, Eq. 6 12: 14.9, 8: 15.3 / 17.5).
int level_cluster(int variant, const Grid3* g, int n) {
    const ActiveClusters* active = active_clusters();
    int best_c = kLevelCluster / 2;
    double best = 1e30;
    for (int C = 1; active && C <= kLevelCluster; ++C) {
        if (active->n[C] < 1) continue;
        int tile = 0;
        for (int j = 0; j < n && tile >= 0; ++j) {
            if (j > 0 && g[j].nx == g[j - 1].nx && g[j].ny == g[j - 1].ny && g[j].nz == g[j - 1].nz)
                continue;
            int tr, tp, smem;
            if (level_tiles(g[j], variant, C, &tr, &tp, &smem))
                tile = std::max(tile, tr * tp * g[j].nx);
            else
                tile = -1;  // does not fit
        }
        if (tile < 0) continue;
        const int turns = (n + active->n[C] - 1) / active->n[C];
        const double us = turns * (1.6 + 0.04 * C + 0.002 * tile);
        if (us < best) {
            best = us;
            best_c = C;
        }
    }
    return best_c;
}

bool level_resident(int variant, const Grid3& g) {
    int tr, tp, smem;
    return (long long)g.nx * g.ny * g.nz <= kLevelMaxVoxels &&
           level_tiles(g, variant, kLevelCluster / 2, &tr, &tp, &smem) && active_clusters();
}

bool level_group_add(LevelGroup& G, int variant, const LevelArgs& a) {
    if (G.n >= kGroupMax || G.cluster < 1 || G.cluster > kLevelCluster) return false;
    int smem;
    LevelArgs& b = G.a[G.n];
    b = a;
    if (!level_tiles(a.g, variant, G.cluster, &b.tile_rows, &b.tile_planes, &smem)) return false;
    G.smem = std::max(G.smem, smem);
    G.n += 1;
    return true;
}

cudaError_t launch_level(int variant, int img_type, const LevelGroup& G, cudaStream_t s) {
    if (G.n < 1) return cudaErrorInvalidValue;
    if (img_type == kStoreF32) return launch_level_types<float>(variant, G, G.smem, s);
    if (img_type == kStoreI16) return launch_level_types<int16_t>(variant, G, G.smem, s);
    return cudaErrorInvalidValue;
}

}  // namespace dirk
