// Grids of the transpose tile (x = A^T y, Sec. 1, Eq. 1 read column-wise):
// one kernel per launch configuration (DevGeom::bwd_config), storage type
// and output layout, instantiated by transpose_zfast.cu (padded z-fastest
// output, the solvers' layout) and transpose_abi.cu (x[k][j][i]), which
// compile in parallel.
//
// PASSES selects the kernel that sums a block of angles [a_begin, a_end)
// with FP32 running sums kept between passes (launch_backward); the
// single-pass kernel sums every angle and takes neither the angle range nor
// the running-sum buffers (fewer live registers through the angle loop).
#pragma once

#include "patch_tile.cuh"

namespace cbct {

// Tiles of 2 or 4 voxels per lane run 3 CTAs per SM (80 registers): the
// 2-voxel tiles clip their detector columns across the lanes, which measured
// 36.6 ms at 256^3 this way against 39.0 ms at 4 CTAs.
template <typename T, bool ZFAST, int CX, int K, bool PASSES>
__global__ void __launch_bounds__(BWD_THREADS, K >= 2 ? 3 : 4)
backward_kernel(DevGeom g, const float *__restrict__ proj, T *__restrict__ vol, Epilogue epi, int a_begin, int a_end,
                const float *acc_in, float *acc_out) {
    if (epi.stop && *epi.stop) return;
    auto partial_at = [&]() -> double * {
        const size_t b = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        return epi.partial ? epi.partial + b * TILE_PARTIALS : nullptr;
    };
    if (PASSES)
        backward_tile<T, ZFAST, CX, K>(g, proj, vol, epi, blockIdx.x, blockIdx.y, blockIdx.z, a_begin, a_end, acc_in,
                                       acc_out, partial_at);
    else
        backward_tile<T, ZFAST, CX, K>(g, proj, vol, epi, blockIdx.x, blockIdx.y, blockIdx.z, 0, g.nangles, nullptr,
                                       nullptr, partial_at);
}

// Patch tiles.  32 warps per SM (64 registers): A^T y at 256^3 / 512^2 / 90
// angles 2.80 ms, with 24 warps (80 registers) 3.07 ms; four voxels per lane
// take 20 % fewer instructions but leave 16 warps and measured 3.13 ms.
template <typename T, bool ZFAST, int PATCHES, bool ALONG_X, int ZG, int SPLITS, bool PASSES>
__global__ void __launch_bounds__(BWD_THREADS, 4)
patch_kernel(DevGeom g, const float *__restrict__ proj, T *__restrict__ vol, Epilogue epi, int a_begin, int a_end,
             const float *acc_in, float *acc_out) {
    extern __shared__ float4 patch_lists[];
    if (epi.stop && *epi.stop) return;
    auto partial_at = [&]() -> double * {
        const size_t b = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        return epi.partial ? epi.partial + b * TILE_PARTIALS : nullptr;
    };
    if (PASSES)
        patch_tile<T, ZFAST, PATCHES, ALONG_X, ZG, SPLITS>(g, proj, vol, epi, blockIdx.x, blockIdx.y, blockIdx.z, a_begin,
                                                  a_end, acc_in, acc_out, partial_at, (char *)patch_lists);
    else
        patch_tile<T, ZFAST, PATCHES, ALONG_X, ZG, SPLITS>(g, proj, vol, epi, blockIdx.x, blockIdx.y, blockIdx.z, 0, g.nangles,
                                                  nullptr, nullptr, partial_at, (char *)patch_lists);
}

template <typename T, bool ZF, bool PASSES>
void launch_backward_tp(const DevGeom &g, const float *y, void *x, const Epilogue &epi, cudaStream_t s, int a0,
                        int a1, const float *acc_in, float *acc_out) {
    const dim3 grid = backward_grid(g);
    T *xx = (T *)x;
    if (backward_patches(g)) {
#define CBCT_PATCH(PATCHES, ALONG_X, ZG, SPLITS)                                                               \
    patch_kernel<T, ZF, PATCHES, ALONG_X, ZG, SPLITS, PASSES>                                                  \
        <<<grid, BWD_THREADS, patch_shared_bytes<PATCHES, ZG, SPLITS>(g.patch_columns), s>>>(g, y, xx, epi, a0, a1, \
                                                                                             acc_in, acc_out)
        switch (g.bwd_config) {     // patches x stacks of 64 voxels x angle ranges
        case 1:
        case 3:
            if (g.patch_single)
                CBCT_PATCH(1, false, 1, 8);
            else if (g.bwd_config == 1)
                CBCT_PATCH(2, true, 1, 4);
            else
                CBCT_PATCH(2, false, 1, 4);
            break;
        case 4: CBCT_PATCH(2, true, 2, 2); break;
        case 5: CBCT_PATCH(2, false, 2, 2); break;
        case 6: CBCT_PATCH(2, true, 4, 1); break;
        default: CBCT_PATCH(2, false, 4, 1); break;
        }
#undef CBCT_PATCH
        return;
    }
#define CBCT_BWD(CX, K) \
    backward_kernel<T, ZF, CX, K, PASSES><<<grid, BWD_THREADS, 0, s>>>(g, y, xx, epi, a0, a1, acc_in, acc_out)
    switch (g.bwd_config) {         // shapes as in backward_shape
    case 1: CBCT_BWD(4, 2); break;
    case 2: CBCT_BWD(8, 1); break;
    case 3: CBCT_BWD(2, 2); break;
    case 4: case 6: case 9: CBCT_BWD(4, 4); break;
    case 5: case 7: case 8: CBCT_BWD(2, 4); break;
    default: CBCT_BWD(4, 1); break;
    }
#undef CBCT_BWD
}

// One launch over angles [a0, a1) in storage type t; the single-pass kernel
// when the launch covers every angle with no running sums.
template <bool ZF>
void launch_backward_layout(const DevGeom &g, const float *y, void *x, cbct_dtype t, const Epilogue &epi,
                            cudaStream_t s, int a0, int a1, const float *acc_in, float *acc_out) {
    const bool passes = acc_in || acc_out || a0 != 0 || a1 != g.nangles;
    switch (t) {
    case CBCT_F32:
        passes ? launch_backward_tp<float, ZF, true>(g, y, x, epi, s, a0, a1, acc_in, acc_out)
               : launch_backward_tp<float, ZF, false>(g, y, x, epi, s, a0, a1, acc_in, acc_out);
        break;
    case CBCT_F16:
        passes ? launch_backward_tp<__half, ZF, true>(g, y, x, epi, s, a0, a1, acc_in, acc_out)
               : launch_backward_tp<__half, ZF, false>(g, y, x, epi, s, a0, a1, acc_in, acc_out);
        break;
    case CBCT_BF16:
        passes ? launch_backward_tp<__nv_bfloat16, ZF, true>(g, y, x, epi, s, a0, a1, acc_in, acc_out)
               : launch_backward_tp<__nv_bfloat16, ZF, false>(g, y, x, epi, s, a0, a1, acc_in, acc_out);
        break;
    }
}

}  // namespace cbct
