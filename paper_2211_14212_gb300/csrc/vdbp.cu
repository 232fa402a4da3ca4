// Voxel-driven, interpolating backprojector: the usual fast approximation of
// A^T that is not its exact transpose, the kind of backprojector AB-/BA-GMRES
// are meant for (Sec. 2.1.4).  Every voxel centre is projected onto every
// detector and the projection is sampled there by bilinear interpolation
// (zero outside the detector), weighted by the expected sum of A's entries of
// the rays through the voxel,
//     w = dx dy dz mag^2 |d'| / (du dv DSD),   mag = DSD / (DSO - <c, s_hat>),
// with |d'| the source-to-pixel distance of the sampled point.
//
// Work layout as the exact transpose's gather: a warp owns one voxel column
// (i, j) and 32 K voxels along z (lane l: k0 + kk 32 + l); the neighbouring rows
// of its lanes make the v-fastest projection reads contiguous.
// The column's projected u, magnification and weights of an angle are the same
// for all its voxels: the lanes work them out for 32 angles at once (with the
// IEEE divisions), and the walk over the angles reads them back from shared
// memory.  It was bound by instruction issue, most of it these divisions and
// the square root repeated by every lane.  BA-GMRES, 4 iterations (5 products
// with this kernel), 128^3 / 256^2 / 180 angles: 10.7 -> 7.8 ms.
#include <cmath>

#include "common.cuh"

namespace cbct {

constexpr int VD_CX = 4, VD_CY = 2, VD_THREADS = 256;

// One angle of a voxel column: weights of its two detector columns (voxel
// volume, mag^2 and the horizontal interpolation), mag / dv, their offsets
// within the projection, mag^2 and DSD^2 + u^2; valid: bit 0 / 1 set if the first
// / second column lies on the detector.
struct VdAngle {
    float w0, w1, rows, mag2, c;
    unsigned col0, col1, valid;
};

// Voxels per lane: 4 above 64 slices (the walk's share per angle halves), 2
// below (4 would leave half the lanes idle).
template <bool ZFAST, int K>
__global__ void __launch_bounds__(VD_THREADS)
voxel_backproject_kernel(DevGeom g, const float *__restrict__ proj, float *__restrict__ vol) {
    __shared__ VdAngle table[VD_THREADS / 32][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * VD_CX + (warp % VD_CX), j = blockIdx.y * VD_CY + (warp / VD_CX);
    const int k0 = blockIdx.z * 32 * K;
    if (i >= g.nx || j >= g.ny) return;               // uniform across the warp
    const float xc = g.bx0 + (i + 0.5f) * g.dx, yc = g.by0 + (j + 0.5f) * g.dy;
    const float cu = 0.5f * (g.nu - 1), cv = 0.5f * (g.nv - 1);
    const float wvol = g.dx * g.dy * g.dz / (g.du * g.dv * g.dsd);
    float zc[K], acc[K];
#pragma unroll
    for (int kk = 0; kk < K; ++kk) {
        zc[kk] = g.bz0 + (k0 + kk * 32 + lane + 0.5f) * g.dz;
        acc[kk] = 0.0f;
    }
    // largest |z| of the warp's voxels: bounds their rows
    const float zlo = g.bz0 + (k0 + 0.5f) * g.dz, zhi = g.bz0 + (k0 + 32 * K - 0.5f) * g.dz;
    const float zmax = fmaxf(fabsf(zlo), fabsf(zhi));
    const size_t nuv = (size_t)g.nu * g.nv;
    for (int a0 = 0; a0 < g.nangles; a0 += 32) {
        bool hit = false;
        if (a0 + lane < g.nangles) {
            const float2 cs = __ldg(&g.trig[a0 + lane]);
            const float mag = g.dsd / (g.dso - (xc * cs.x + yc * cs.y));
            const float u = (-xc * cs.y + yc * cs.x) * mag;
            const float fu = u / g.du + cu;
            const float fu0 = floorf(fu);
            const int iu = (int)fu0;
            const float tu = fu - fu0;
            hit = iu >= -1 && iu < g.nu;              // otherwise the column projects off the detector
            const float wmag = wvol * mag * mag;
            VdAngle t;
            t.w0 = wmag * (1.0f - tu);
            t.w1 = wmag * tu;
            t.rows = mag / g.dv;
            t.mag2 = mag * mag;
            t.c = g.dsd * g.dsd + u * u;
            t.col0 = (unsigned)min(max(iu, 0), g.nu - 1) * (unsigned)g.nv;
            t.col1 = (unsigned)min(max(iu + 1, 0), g.nu - 1) * (unsigned)g.nv;
            t.valid = (iu >= 0 ? 1u : 0u) | (iu + 1 < g.nu ? 2u : 0u);
            table[warp][lane] = t;
        }
        const unsigned hits = __ballot_sync(0xffffffffu, hit);
        __syncwarp();
        const int n = min(32, g.nangles - a0);
        const float *pa = proj + (size_t)a0 * nuv;
        for (int s = 0; s < n; ++s, pa += nuv) {
            if (!(hits >> s & 1)) continue;
            const VdAngle t = table[warp][s];
            const float *p0 = pa + t.col0, *p1 = pa + t.col1;
            auto add = [&](int kk, float y00, float y01, float y10, float y11, float tv) {
                const float lo = __fmaf_rn(t.w1, y10, t.w0 * y00), hi = __fmaf_rn(t.w1, y11, t.w0 * y01);
                const float val = __fmaf_rn(tv, hi, (1.0f - tv) * lo);
                float len;
                asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(len) : "f"(__fmaf_rn(zc[kk] * zc[kk], t.mag2, t.c)));
                acc[kk] = __fmaf_rn(len, val, acc[kk]);
            };
            if (t.valid == 3 && __fmaf_rn(zmax, t.rows, 2.0f) <= cv) {    // the warp samples inside the detector only
#pragma unroll
                for (int kk = 0; kk < K; ++kk) {
                    const float fv = __fmaf_rn(zc[kk], t.rows, cv), fv0 = floorf(fv);
                    const int iv = (int)fv0;
                    add(kk, __ldg(p0 + iv), __ldg(p0 + iv + 1), __ldg(p1 + iv), __ldg(p1 + iv + 1), fv - fv0);
                }
            } else {
#pragma unroll
                for (int kk = 0; kk < K; ++kk) {
                    const float fv = __fmaf_rn(zc[kk], t.rows, cv), fv0 = floorf(fv);
                    const int iv = (int)fv0;
                    const bool v0 = iv >= 0 && iv < g.nv, v1 = iv + 1 >= 0 && iv + 1 < g.nv;
                    const bool u0 = t.valid & 1, u1 = t.valid & 2;      // zero outside
                    add(kk, u0 && v0 ? __ldg(p0 + iv) : 0.0f, u0 && v1 ? __ldg(p0 + iv + 1) : 0.0f,
                        u1 && v0 ? __ldg(p1 + iv) : 0.0f, u1 && v1 ? __ldg(p1 + iv + 1) : 0.0f, fv - fv0);
                }
            }
        }
        __syncwarp();                                  // the table is rewritten
    }
#pragma unroll
    for (int kk = 0; kk < K; ++kk) {
        const int k = k0 + kk * 32 + lane;
        if (k >= g.nz) continue;
        const size_t vi = ZFAST ? (size_t)(zf_col(g, i, j) + k) : ((size_t)k * g.ny + j) * g.nx + i;
        vol[vi] = acc[kk];
    }
}

template <int K>
static void launch_voxel_backproject_k(const DevGeom &g, const float *y_vfast, float *x, bool zfast, cudaStream_t s) {
    const dim3 grid((g.nx + VD_CX - 1) / VD_CX, (g.ny + VD_CY - 1) / VD_CY, (g.nz + 32 * K - 1) / (32 * K));
    if (zfast)
        voxel_backproject_kernel<true, K><<<grid, VD_THREADS, 0, s>>>(g, y_vfast, x);
    else
        voxel_backproject_kernel<false, K><<<grid, VD_THREADS, 0, s>>>(g, y_vfast, x);
}

cbct_status launch_voxel_backproject(const DevGeom &g, const float *y_vfast, float *x, bool zfast, cudaStream_t s) {
    if (g.nz > 64)
        launch_voxel_backproject_k<4>(g, y_vfast, x, zfast, s);
    else
        launch_voxel_backproject_k<2>(g, y_vfast, x, zfast, s);
    CBCT_CUDA_TRY(cudaGetLastError());
    return CBCT_OK;
}

}  // namespace cbct

using namespace cbct;

extern "C" cbct_status cbct_backproject_voxel_driven(const cbct_geometry *g, const float *y, float *x,
                                                     cbct_stream stream) {
    if (!g || !y || !x) { set_error("cbct_backproject_voxel_driven: null argument"); return CBCT_EINVAL; }
    const cbct_status dst = require_geometry_device(g, "cbct_backproject_voxel_driven");
    if (dst != CBCT_OK) return dst;
    cudaStream_t s = (cudaStream_t)stream;
    float *tmp = nullptr;
    CBCT_CUDA_TRY(cudaMallocAsync(&tmp, (size_t)cbct_geometry_num_rays(g) * sizeof(float), s));
    cbct_status st = launch_proj_relayout(g->dev, y, tmp, CBCT_F32, true, s);
    if (st == CBCT_OK) st = launch_voxel_backproject(g->dev, tmp, x, false, s);
    cudaFreeAsync(tmp, s);
    return st;
}
