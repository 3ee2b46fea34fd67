// dir_xy.cuh -- the x and y passes of the Gaussian (Sec. 2.5) as warps that
// march down y: out = G_y * G_x * in, plane by plane, radius 3.
//
// A warp owns a strip: 32 columns x its output rows x 4 planes of one
// component, 8 lanes per plane with 4 adjacent columns each.  Rows arrive in
// boxes of 7 (two in flight per warp) by TMA; per row a lane reads the 12
// floats around its columns, filters them in x (28 multiply-adds), keeps the
// last 7 filtered rows in registers and filters those in y on packed pairs (14
// multiply-adds for 4 outputs).  Seven rows per box make the register ring
// rotate by renaming.  Warps share nothing, so there is no block barrier and
// no exchange through shared memory between the passes; a strip redoes the x
// pass of 6 halo rows, which is what its length is chosen against.
//
// Taps oldest first, fused multiply-adds from zero, as smooth2_kernel: the
// same output bit for bit.
//
// The form it replaces on large levels (32-row tiles of 256 threads, rows
// exchanged through shared memory between the passes behind two barriers per
// plane) issued 145 warp instructions per 32 voxels and kept the shared-memory
// pipe 81 % busy: 39.0 us at 256x256x100 and 199 us at 512x512x160 for 24 B per
// voxel; the strips take 30.0 us and 151 us (6.66 TB/s, the copy rate).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "dir_common.cuh"
#include "dir_launch.h"
#include "dir_pair.cuh"
#include "dir_stencil.cuh"

namespace dirk {

constexpr int XYR = 3;                    // radius
constexpr int XYW = 32, XYP = 4;          // strip width and planes
constexpr int XYB = 2 * XYR + 1;          // rows per box (= ring length)
constexpr int XYWB = XYW + 8;             // box width, x halo 16-byte aligned
constexpr int XYBOX = XYP * XYB * XYWB * 4;  // bytes of a box: [XYP][XYB][XYWB] floats
constexpr int XYWARPS = 4;                // warps per block
constexpr int XYSTAGES = 2;
constexpr int XYSMEM = 128 + XYWARPS * XYSTAGES * XYBOX;
static_assert(XYBOX % 128 == 0, "boxes stay 128-byte aligned");

// Output rows of a strip of nb boxes
__host__ __device__ constexpr int xy_rows(int nb) { return XYB * nb - 2 * XYR; }

// The strips of a volume: tiles along x fastest, then strips along y, then
// components, then groups of planes (bottom up, so that the z + force kernel,
// which walks top down, finds the last ones in L2)
struct XYStrips {
    int nb;     // boxes per strip
    int tx, cy; // tiles along x, strips along y
    int n;      // strips
    __host__ __device__ int blocks() const { return (n + XYWARPS - 1) / XYWARPS; }
};
inline XYStrips xy_strips(const Grid3& g, int nb) {
    XYStrips s;
    s.nb = nb;
    s.tx = (g.nx + XYW - 1) / XYW;
    s.cy = (g.ny + xy_rows(nb) - 1) / xy_rows(nb);
    s.n = s.tx * s.cy * 3 * ((g.nz + XYP - 1) / XYP);
    return s;
}
// Strips or tiles: strips where the shortest ones number 16 warps per SM. Below
// that the tiles' shorter chain wins. Measured per passive iteration, tiles ->
// strips: 96x96x48 (1,296 strips) 11.9 -> 14.1 us, 128x128x25 (1,344) 12.3 ->
// 14.4, 128x128x50 (2,496) 14.9 -> 14.4, 128x128x64 (3,072) 19.9 -> 18.4,
// 193x171x87 55.2 -> 46.4, 256x256x100 83.4 -> 76.4, 512x512x160 505 -> 456.
inline bool xy_use_strips(const Grid3* g, int n, int num_sms) {
    long long strips = 0;
    for (int j = 0; j < n; ++j) strips += xy_strips(g[j], 2).n;
    return strips >= 16LL * num_sms;
}
// Boxes per strip: the shortest strips that are all resident at once (slots:
// resident warps), so that none waits for a second wave; volumes with too many
// take 4 boxes, where neighbouring strips' halo rows still meet in L2.
// Measured, all strips of a launch alone: 256x256x100 7 boxes 30.0 us (2: 32.8,
// 4: 30.5), 193x171x87 5 boxes 14.4 us (3: 16.4, 8: 18.5), 512x512x160 4 boxes
// 151 us (2: 169, 7: 161).
inline int xy_strip_boxes(const Grid3* g, int n, long long slots) {
    for (int nb = 2; nb <= 7; ++nb) {
        long long strips = 0;
        for (int j = 0; j < n; ++j) strips += xy_strips(g[j], nb).n;
        if (strips <= slots) return nb;
    }
    return 4;
}

// One strip: tile column tx, strip row cy (of strips of nb boxes), component
// comp, planes 4 zg .. 4 zg + 3.  slots, bars: this warp's own.
__device__ __forceinline__ void xy_strip(const CUtensorMap* map, const SmoothArgs& a, int nb, int tx,
                                         int cy, int comp, int zg, float* slots, uint64_t* bars) {
    constexpr int R = XYR, K = 2 * R + 1;
    const Grid3 g = a.g;
    const int lane = threadIdx.x & 31, sub = lane >> 3, gq = lane & 7;
    const int x0 = tx * XYW, y0 = cy * xy_rows(nb), z0 = zg * XYP;
    const int y1 = min(y0 + xy_rows(nb), g.ny);
    const int boxes = (y1 - y0 + 2 * R + XYB - 1) / XYB;
    const int bx = x0 - 4;
    auto issue = [&](int b) {
        uint64_t* bar = &bars[b % XYSTAGES];
        fence_proxy_async();
        mbar_arrive_expect_tx(bar, (uint32_t)XYBOX);
        tma_load_4d(slots + (b % XYSTAGES) * (XYBOX / 4), map, bx, y0 - R + XYB * b, z0, comp, bar);
    };
    if (lane == 0) {
        for (int s = 0; s < XYSTAGES; ++s) mbar_init(&bars[s], 1);
        fence_mbar_init();
        pdl_wait();
        for (int b = 0; b < XYSTAGES && b < boxes; ++b) issue(b);
    }
    pdl_wait();  // every lane: out is written below, which the kernel before reads
    __syncwarp();

    const bool edge = bx < 0 || bx + XYWB > g.nx;
    const int x = x0 + 4 * gq, z = z0 + sub;
    const int nstore = z < g.nz ? min(g.nx - x, 4) : 0;  // columns this lane stores
    // output row of input row y0 - R + 7 b + r is R rows before it
    float* o = static_cast<float*>(a.out) + (size_t)comp * g.cs +
               ((long long)x + (long long)g.px * (y0 - 2 * R) + g.plane * z);
    f32x2 ring[K][2];
#pragma unroll
    for (int t = 0; t < K; ++t) ring[t][0] = ring[t][1] = 0ull;
    for (int b = 0; b < boxes; ++b) {
        float* slot = slots + (b % XYSTAGES) * (XYBOX / 4);
        const bool ok = mbar_wait_bounded(&bars[b % XYSTAGES], (uint32_t)((b / XYSTAGES) & 1),
                                          kWaitLimitNs);
        if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0 && a.err) atomicOr(a.err, kErrTmaTimeout);
            return;
        }
        if (edge) {  // replicate the columns outside the volume, a lane per row
            if (lane < XYP * XYB) {
                float* r = slot + lane * XYWB;
                if (bx < 0) {
                    const float left = r[4];
                    r[1] = r[2] = r[3] = left;
                }
                const int hi = g.nx - bx;
                if (hi < XYWB) {
                    const float right = r[hi - 1];
                    for (int j = hi; j < min(hi + R, XYWB); ++j) r[j] = right;
                }
            }
            __syncwarp();
        }
        const float* row = slot + sub * (XYB * XYWB) + 4 * gq;
        const int ytop = y0 - R + XYB * b;   // input row of the box's first row
        const int first = b == 0 ? R - y0 : 0;  // box row of y = 0, where above it none exist
#pragma unroll
        for (int r = 0; r < XYB; ++r) {
            if (ytop + r < g.ny) {
                const float4* src =
                    reinterpret_cast<const float4*>(row + (r < R ? max(r, first) : r) * XYWB);
                const float4 p = src[0], q = src[1], s = src[2];
                const float in[12] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w, s.x, s.y, s.z, s.w};
                float f[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    f[j] = 0.0f;
#pragma unroll
                    for (int t = 0; t < K; ++t)
                        f[j] = fmaf(a.taps.wf[t <= R ? t : 2 * R - t], in[4 - R + j + t], f[j]);
                }
                ring[r][0] = f2_pack(f[0], f[1]);
                ring[r][1] = f2_pack(f[2], f[3]);
            } else {  // rows past the last: its filtered values again
                ring[r][0] = ring[(r + K - 1) % K][0];
                ring[r][1] = ring[(r + K - 1) % K][1];
            }
            if ((b > 0 || r == K - 1) && ytop + r - R < y1) {
                f32x2 v0 = 0ull, v1 = 0ull;
#pragma unroll
                for (int t = 0; t < K; ++t) {
                    const float2 w2 = a.taps.wp[t <= R ? t : 2 * R - t];
                    const f32x2 w = f2_pack(w2.x, w2.y);
                    v0 = f2_fma(w, ring[(r + 1 + t) % K][0], v0);
                    v1 = f2_fma(w, ring[(r + 1 + t) % K][1], v1);
                }
                float4 v;
                f2_unpack(v0, v.x, v.y);
                f2_unpack(v1, v.z, v.w);
                if (nstore == 4) {
                    *reinterpret_cast<float4*>(o) = v;
                } else if (nstore > 0) {
                    o[0] = v.x;
                    if (nstore > 1) o[1] = v.y;
                    if (nstore > 2) o[2] = v.z;
                }
            }
            o += g.px;
        }
        __syncwarp();  // every lane has read the slot before it is filled again
        if (lane == 0 && b + XYSTAGES < boxes) issue(b + XYSTAGES);
    }
}

// The strips of block `block` of a volume's launch, one per warp.
__device__ __forceinline__ void xy_strip_block(const CUtensorMap* map, const SmoothArgs& a,
                                               const XYStrips& st, int block) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint64_t bars[XYWARPS][XYSTAGES];
    if (a.stop_iter != nullptr && *a.stop_iter < a.iter) return;
    unsigned char* base = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    const int w = threadIdx.x >> 5;
    const unsigned u = (unsigned)block * XYWARPS + w;
    pdl_trigger();
    if (u >= (unsigned)st.n) return;
    const unsigned q = u / (unsigned)st.tx, tx = u % (unsigned)st.tx;
    const unsigned q2 = q / (unsigned)st.cy, cy = q % (unsigned)st.cy;
    xy_strip(map, a, st.nb, tx, cy, q2 % 3, q2 / 3,
             reinterpret_cast<float*>(base) + w * XYSTAGES * (XYBOX / 4), bars[w]);
}

inline bool make_xy_strip_map(CUtensorMap* map, const void* ptr, const Grid3& g) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    const cuuint64_t dims[4] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz, 3};
    const cuuint64_t strides[3] = {(cuuint64_t)g.px * 4, (cuuint64_t)g.plane * 4,
                                   (cuuint64_t)g.cs * 4};
    const cuuint32_t box[4] = {(cuuint32_t)XYWB, (cuuint32_t)XYB, (cuuint32_t)XYP, 1u};
    const cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void*>(ptr), dims, strides, box,
               estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace dirk
