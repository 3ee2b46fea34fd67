// dir_force_d.cu -- kernels and launchers of the Eqs. (3)-(6) split iteration
// with the difference image formed once per voxel (block functions in
// dir_split_d.cuh): the z + D pass and the stencil force pass.
#include <cuda.h>
#include <cuda_runtime.h>

#include "dir_split_d.cuh"

namespace dirk {

template <int V, int FTZ, typename TI, bool UW>
__global__ void __launch_bounds__(FNT, UW || V == 5 ? 4 : 5)
    force_zd_kernel(const __grid_constant__ CUtensorMap tmap, const ForceArgs a, const Taps taps) {
    zd_block<V, FTZ, TI, UW>(&tmap, a, taps, BlockPos::of_grid());
}

template <int V, int FTZ, typename TI, bool UW>
__global__ void __launch_bounds__(FNT, UW ? 4 : 3)
    force_st_kernel(const __grid_constant__ CUtensorMap dmap,
                    const __grid_constant__ CUtensorMap smap,
                    const __grid_constant__ CUtensorMap tmap,
                    const __grid_constant__ CUtensorMap emap, const ForceArgs a, const Taps taps) {
    st_block<V, FTZ, TI, UW>(&dmap, &smap, &tmap, &emap, a, taps, BlockPos::of_grid());
}

namespace {

// 4-D tiled map over a pitched volume of ncomp components (esz-byte elements)
bool map4(CUtensorMap* m, CUtensorMapDataType t, const void* p, const Grid3& g, int ncomp, int esz,
          int bx, int by, int bz) {
    EncodeTiledFn enc = encode_fn();
    if (!enc || p == nullptr) return false;
    const cuuint64_t dims[4] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz,
                                (cuuint64_t)ncomp};
    const cuuint64_t str[3] = {(cuuint64_t)g.px * esz, (cuuint64_t)g.plane * esz,
                               (cuuint64_t)g.cs * esz};
    const cuuint32_t box[4] = {(cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bz, (cuuint32_t)ncomp};
    const cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
    return enc(m, t, 4, const_cast<void*>(p), dims, str, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

dim3 brick_grid(const Grid3& g, int ftz) {
    return dim3((g.nx + FTX - 1) / FTX, (g.ny + FTY - 1) / FTY, (g.nz + ftz - 1) / ftz);
}

template <int V, int FTZ, typename TI, bool UW>
cudaError_t launch_zd(const ForceArgs& a, const Taps& taps, cudaStream_t s) {
    using Z = ZDGeom<FTZ>;
    CUtensorMap tmap;
    if (!map4(&tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, a.u, a.g, 3, 4, FTX, FTY, Z::NPZ))
        return cudaErrorInvalidValue;
    static KernelSetup setup;  // per instantiation
    const cudaError_t e = setup_kernel(setup, force_zd_kernel<V, FTZ, TI, UW>, Z::SMEM);
    if (e != cudaSuccess) return e;
    return launch_ex(force_zd_kernel<V, FTZ, TI, UW>, brick_grid(a.g, FTZ), dim3(FTX, FTY, 1),
                     Z::SMEM, s, a.pdl, tmap, a, taps);
}

template <int V, int FTZ, typename TI, bool UW>
cudaError_t launch_st(const ForceArgs& a, const Taps& taps, cudaStream_t s) {
    using F = STGeom<FTZ, V, TI, UW>;
    CUtensorMap dmap, smap, tmap, emap;
    if (!map4(&dmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, a.dbuf, a.g, 1, 4, F::DW, F::DH, F::DD) ||
        !map4(&smap, tma_type<TI>(), a.S, a.g, 1, (int)sizeof(TI), F::FSW, FSH, F::DD) ||
        !map4(&tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, a.u, a.g, 3, 4, FTX, FTY, F::NPZ))
        return cudaErrorInvalidValue;
    if (F::IC) {
        if (!map4(&emap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, a.dbuf2, a.g, 1, 4, FTX, FTY, FTZ))
            return cudaErrorInvalidValue;
    } else {
        emap = tmap;  // not read
    }
    static KernelSetup setup;  // per instantiation
    const cudaError_t e = setup_kernel(setup, force_st_kernel<V, FTZ, TI, UW>, F::SMEM);
    if (e != cudaSuccess) return e;
    return launch_ex(force_st_kernel<V, FTZ, TI, UW>, brick_grid(a.g, FTZ), dim3(FTX, FTY, 1),
                     F::SMEM, s, a.pdl, dmap, smap, tmap, emap, a, taps);
}

template <int V, typename TI>
cudaError_t launch_d_pair(const ForceArgs& zd, const ForceArgs& st, const Taps& taps,
                          cudaStream_t s) {
    if (st.u != zd.v) {  // u formed again: bricks of 4 (z + D), 4 or 8 planes
        const cudaError_t e = launch_zd<V, 4, TI, false>(zd, taps, s);
        if (e != cudaSuccess) return e;
        return st.depth >= 8 ? launch_st<V, 8, TI, false>(st, taps, s)
                             : launch_st<V, 4, TI, false>(st, taps, s);
    }
    cudaError_t e = cudaErrorInvalidValue;
    switch (zd.depth) {
        case 8:
        case 6:
        case 4: e = launch_zd<V, 4, TI, true>(zd, taps, s); break;
        case 2: e = launch_zd<V, 2, TI, true>(zd, taps, s); break;
        case 1: e = launch_zd<V, 1, TI, true>(zd, taps, s); break;
        default: break;
    }
    if (e != cudaSuccess) return e;
    switch (st.depth) {
        case 8: return launch_st<V, 8, TI, true>(st, taps, s);
        case 6:
        case 4: return launch_st<V, 4, TI, true>(st, taps, s);
        case 2: return launch_st<V, 2, TI, true>(st, taps, s);
        case 1: return launch_st<V, 1, TI, true>(st, taps, s);
        default: return cudaErrorInvalidValue;
    }
}

template <typename TI>
cudaError_t launch_d_types(int variant, const ForceArgs& zd, const ForceArgs& st,
                           const Taps& taps, cudaStream_t s) {
    switch (variant) {
        case 2: return launch_d_pair<2, TI>(zd, st, taps, s);
        case 3: return launch_d_pair<3, TI>(zd, st, taps, s);
        case 4: return launch_d_pair<4, TI>(zd, st, taps, s);
        case 5: return launch_d_pair<5, TI>(zd, st, taps, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

bool force_d_supported(int variant, const ForceArgs& a, const Taps& taps) {
    return variant >= 2 && variant <= 5 && force_zs_supported(variant, a, taps);
}

// u written by the z + D pass, or formed again by the force pass: written on
// levels of at most 2^20 voxels, whose t, u, D and images stay in L2.  Measured
// per iteration, written -> formed again, Eq. 3 / Eq. 6: 64x64x25 7.95 -> 8.37 /
// 8.36 -> 8.81 us, 128x128x50 18.5 -> 19.9 / 21.2 -> 21.8, 128x128x64 20.6 ->
// 21.1 / 23.6 -> 24.2; above, 160x160x64 28.6 -> 28.2 / 32.9 -> 33.0, 192x192x64
// 39.7 -> 37.1 / 45.3 -> 44.7, 193x171x87 57.1 -> 53.2 / 65.7 -> 64.7,
// 256x256x100 103.2 -> 96.1 / 117.1 -> 114.1.
bool force_d_writes_u(long long voxels) { return voxels <= (1LL << 20); }

int force_d_planes(int variant, bool writes_u) { return (variant == 5 ? 2 : 1) + (writes_u ? 3 : 0); }

// Brick depth of the force pass (the z + D pass caps it at 4): 8 for Eqs. 3-5
// where such bricks number three per SM, else 4 where those number one per SM,
// else 2.  Measured per iteration with the force pass at 2 / 4 / 8, Eq. 3: 48x48x24
// 7.7 / 8.0 / 8.5 us, 64x64x25 7.95 / 7.81 / 8.40, 96x96x48 13.6 / 12.9 / 13.4,
// 128x128x64 21.6 / 20.7 / 19.8.  Eq. 6 stays at 4: with its d box, 8 leaves three
// blocks per SM (128x128x64 23.7 against 23.9; 256x256x100 113.4 against 119).
// Blocks per SM on large levels: five of the z + D kernel for Eqs. 3-5 (95.9 us per
// iteration at 256x256x100 against 97.9 with four), four for Eq. 6 (119 against 122:
// its two interpolations want the registers).
int force_d_depth(int variant, const Grid3& g, int num_sms) {
    const long long bxy = (long long)((g.nx + FTX - 1) / FTX) * ((g.ny + FTY - 1) / FTY);
    if (variant != 5 && bxy * ((g.nz + 7) / 8) >= 3LL * num_sms) return 8;
    return bxy * ((g.nz + 3) / 4) >= num_sms ? 4 : 2;
}

cudaError_t launch_force_d(int variant, const ForceArgs& zd, const ForceArgs& st, const Taps& taps,
                           cudaStream_t s) {
    if (!force_d_supported(variant, zd, taps) || zd.dbuf == nullptr ||
        (variant == 5 && zd.dbuf2 == nullptr))
        return cudaErrorInvalidValue;
    if (zd.img_type == kStoreF32) return launch_d_types<float>(variant, zd, st, taps, s);
    return launch_d_types<int16_t>(variant, zd, st, taps, s);
}

}  // namespace dirk
