// Patch tile of the transpose A^T y: a warp sums 2 x 2 voxel columns x 64
// voxels along z (two per lane), angle by angle, in registers.
//
// What bounds a gather here is instruction issue and the L1 wavefronts of the
// projection reads, so the tile shares both as widely as the geometry allows:
//
// - Lists.  The detector columns that cross a patch at an angle and the alpha
//   interval [ain, aout] each of them spends in each of the 4 cells do not
//   depend on z.  The ZG warps that stack up along z over one patch build them
//   together, PT_ANGLES angles at a time, one (detector column, cell) pair per
//   lane, into shared memory.
// - Rows.  Every detector row is assigned to the one slab k in which it leaves
//   the patch (at the far corner's depth): a voxel's rows are consecutive, and
//   the voxels of a column share none.  A row is summed once, with the full
//   length aout - ain, and the sum over a voxel's rows serves all cells of the
//   patch that the detector column crosses.
// - Crossings.  Rays only move away from the mid-plane, so a row that enters
//   its slab k inside the patch does so through the plane nearer to the
//   mid-plane, and spends the part of [ain, aout] before that crossing in the
//   neighbouring slab.  That part is summed apart (D, only the first row of a
//   voxel can have one: the rows that a plane passes between the patch's near
//   and far depth are at most one, PT_MARGIN included, or two in the general
//   walk) and moved from voxel to voxel once, after the last angle.  D is a
//   small part of the sum, so nothing cancels.
//
// Geometries outside patch_columns()'s bounds (steep cones, voxels that cover
// very many detector columns) take backward_tile.
#pragma once

#include "projector_device.cuh"

namespace cbct {

constexpr int PT_ANGLES = 8;             // angles per list
constexpr int PT_STEP = 8;               // detector columns listed in one step of a warp (x 4 cells)
constexpr int PT_MAX_COLUMNS = 24;       // most detector columns across a patch
constexpr float PT_MARGIN = 0.05f;       // pixels; covers the windows' rounding (about 1e-4)
constexpr float PT_NEVER = -FLT_MAX;     // crossing alpha of a row that enters its slab before the patch

// Columns of one angle: mask[s] bit 4 c + q: detector column 8 s + c crosses
// cell q; base: byte offset of the first column within the angle's
// projection; mag: magnification at the far depth; dmag: near minus far.
struct PatchHead {
    unsigned mask[PT_MAX_COLUMNS / PT_STEP], base;
    float mag, dmag, pad[2];
};

// bytes of one patch's two list buffers (columns: DevGeom::patch_columns)
__host__ __device__ __forceinline__ int patch_list_bytes(int columns) {
    return 2 * PT_ANGLES * ((int)sizeof(PatchHead) + columns * 4 * (int)sizeof(float4));
}

__device__ __forceinline__ float fma_sat(float a, float b, float c) { return __saturatef(__fmaf_rn(a, b, c)); }

// First row above plane p (p: planes from the mid-plane, in voxels) at
// magnification `mag`, plus ZMAGIC_BITS.  The margin moves away from the
// mid-plane's side, so that a row assigned beyond the plane has crossed it at
// the far depth, rounding included.
__device__ __forceinline__ float patch_row_offset(float p, float cv) {
    return p > 0.0f ? cv - PT_MARGIN : p < 0.0f ? cv + PT_MARGIN : cv;
}
__device__ __forceinline__ float patch_row(float rows, float mag, float offset) {
    return __fadd_ru(__fmaf_rn(rows, mag, offset), ZMAGIC);
}

// Alpha at which the ray of a row (c: rows from the mid-plane) crosses plane p
// (voxels from the mid-plane): (p rho - c m) / c with rho = dz / dv and
// m = DSO / DSD.  Both are split into a leading part of 11 bits, whose
// products with the half integers p and c are exact, and a remainder, so that
// the difference is rounded at its own size only.
__device__ __forceinline__ float patch_crossing(const DevGeom &g, float c, float p, float p_lo) {
    const float n = __fmaf_rn(p, g.rho_hi, -(c * g.m_hi)) + __fmaf_rn(-c, g.m_lo, p_lo);
    return __fdividef(n, c);
}

// Lists of one angle for the patch at (i0, j0), built by one warp, and the
// crossing parts of the planes at the ends of the block's slabs (edge[0]:
// plane p_edge[0] below, [1]: above; the lanes' sums are per cell lane & 3).
__device__ __forceinline__ void patch_list(const DevGeom &g, const float *__restrict__ wproj, int a, int i0, int j0,
                                           PatchHead *head, float4 *entries, const float (&p_edge)[2],
                                           float (&edge)[2]) {
    const int lane = threadIdx.x & 31;
    const float2 cs = __ldg(&g.trig[a]);
    const float x0 = g.bx0 + i0 * g.dx, x1 = x0 + 2.0f * g.dx;
    const float y0 = g.by0 + j0 * g.dy, y1 = y0 + 2.0f * g.dy;
    float umin = FLT_MAX, umax = -FLT_MAX, magmin = FLT_MAX, magmax = 0.0f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float px = (c & 1) ? x1 : x0, py = (c & 2) ? y1 : y0;
        const float mag = __fdividef(g.dsd, g.dso - (px * cs.x + py * cs.y));
        const float u = (py * cs.x - px * cs.y) * mag;
        umin = fminf(umin, u);
        umax = fmaxf(umax, u);
        magmin = fminf(magmin, mag);
        magmax = fmaxf(magmax, mag);
    }
    const float inv_du = 1.0f / g.du, cu = 0.5f * (g.nu - 1), cv = 0.5f * (g.nv - 1);
    const int iu0 = max(0, (int)ceilf(__fmaf_rn(umin, inv_du, cu - PT_MARGIN)));
    const int iu1 = min(min(g.nu - 1, iu0 + g.patch_columns - 1), (int)floorf(__fmaf_rn(umax, inv_du, cu + PT_MARGIN)));
    const int cell = lane & 3, i = i0 + (cell & 1), j = j0 + (cell >> 1);
    const bool in_volume = i < g.nx && j < g.ny;
    const float dmag = magmax - magmin;
    unsigned mask[PT_MAX_COLUMNS / PT_STEP];
#pragma unroll
    for (int s = 0; s < PT_MAX_COLUMNS / PT_STEP; ++s) {
        mask[s] = 0;
        if (iu0 + s * PT_STEP > iu1) continue;              // uniform
        const int c = s * PT_STEP + (lane >> 2), iu = iu0 + c;
        float ain = -FLT_MAX, aout = FLT_MAX;
        bool miss = !in_volume || iu > iu1;
        if (!miss) {
            const float4 xy = __ldg(&g.ray_xy[(size_t)a * g.nu + iu]);
            const float2 q = __ldg(&g.ray_xyq[(size_t)a * g.nu + iu]);
            clip_slab(RayAxis{xy.x, xy.y, q.x}, g.dx, i, i + 1, ain, aout, miss);
            clip_slab(RayAxis{xy.z, xy.w, q.y}, g.dy, j, j + 1, ain, aout, miss);
        }
        const bool crosses = !miss && ain < aout;
        mask[s] = __ballot_sync(0xffffffffu, crosses);
        if (crosses) {
            const float len = aout - ain, inv = 1.0f / len, start = -ain * inv;
            entries[c * 4 + cell] = make_float4(len, len, inv, start);
            const float *wcol = wproj + ((size_t)a * g.nu + iu) * g.nv;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float p = p_edge[e];
                if (p == 0.0f) continue;                    // no plane to follow at this end
                const float rows = p * g.rho;
                const int first = __float_as_int(patch_row(rows, magmin, patch_row_offset(p, cv))) - ZMAGIC_BITS;
                const int step = p > 0.0f ? 1 : -1;
                int row = p > 0.0f ? first : first - 1;
                const int n = fabsf(rows) * dmag + 2.0f * PT_MARGIN > 1.0f ? 2 : 1;
                for (int t = 0; t < n; ++t, row += step) {
                    if ((unsigned)row >= (unsigned)g.nv) continue;
                    const float at = patch_crossing(g, (float)row - cv, p, p * g.rho_lo);
                    edge[e] = __fmaf_rn(fma_sat(at, inv, start), len * __ldg(wcol + row), edge[e]);
                }
            }
        }
    }
    if (lane == 0) {
        head->mask[0] = mask[0];
        head->mask[1] = mask[1];
        head->mask[2] = mask[2];
        head->base = (unsigned)iu0 * (unsigned)g.nv * 4u;
        head->mag = magmin;
        head->dmag = dmag;
    }
}

// Adds one detector column's part to the cells it crosses (bits of `cells`).
// S: the sum of each voxel's rows, d[t]: its t-th row, at[t]: the alpha at
// which that row enters the voxel's slab.
template <int CAND>
__device__ __forceinline__ void patch_cells(unsigned cells, const float4 *entries, float2 S, const float2 (&d)[CAND],
                                            const float2 (&at)[CAND], float2 (&sum)[4], float2 (&before)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (cells & (1u << q)) {
            const float4 e = entries[q];
            const float2 len = make_float2(e.x, e.y);
            sum[q] = __ffma2_rn(len, S, sum[q]);
#pragma unroll
            for (int t = 0; t < CAND; ++t) {
                const float2 part = make_float2(fma_sat(at[t].x, e.z, e.w), fma_sat(at[t].y, e.z, e.w));
                before[q] = __ffma2_rn(part, __fmul2_rn(len, d[t]), before[q]);
            }
        }
    }
}

// PATCHES patches of 2 x 2 columns side by side (along x if ALONG_X, else
// along y) and ZG stacks of 64 voxels: a tile of PATCHES * ZG warps.
// Angles [a_begin, a_end), running sums and epilogue as in backward_tile.
// lists: PATCHES * patch_list_bytes(g.patch_columns) bytes of shared memory.
template <typename T, bool ZFAST, int PATCHES, bool ALONG_X, int ZG, typename PartialAt>
__device__ __forceinline__ void patch_tile(const DevGeom &g, const float *__restrict__ wproj, T *__restrict__ vol,
                                           const Epilogue &epi, int tx, int ty, int tz, int a_begin, int a_end,
                                           const float *acc_in, float *acc_out, PartialAt &&partial_at, char *lists) {
    constexpr int COLS = PATCHES * 2, SLOTS = 64 * ZG;
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const int patch = warp / ZG, zg = warp % ZG;
    const int i0 = tx * (ALONG_X ? COLS : 2) + (ALONG_X ? 2 * patch : 0);
    const int j0 = ty * (ALONG_X ? 2 : COLS) + (ALONG_X ? 0 : 2 * patch);
    const int kb = tz * SLOTS, k0 = kb + zg * 64;
    const int kend = min(kb + SLOTS, g.nz);
    const float cv = 0.5f * (g.nv - 1), mid = 0.5f * g.nz;
    auto group_sync = [&]() {
        if (ZG == 1)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(1 + patch), "n"(32 * ZG) : "memory");
    };
    char *const mine = lists + patch * patch_list_bytes(g.patch_columns);
    const int entry_stride = g.patch_columns * 4;
    PatchHead *const heads = (PatchHead *)mine;
    float4 *const entries = (float4 *)(mine + 2 * PT_ANGLES * sizeof(PatchHead));

    // planes at the ends of the tile's slabs, when rays cross them outwards
    const float p_edge[2] = {fminf((float)kb - mid, 0.0f), fmaxf((float)kend - mid, 0.0f)};
    float edge[2] = {0.0f, 0.0f};

    // the lane's two voxels
    float zl[2], zu[2], cl[2], cup[2], pp[2], pl[2];
    bool down[2], live[2], middle[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int k = k0 + s * 32 + lane;
        live[s] = k < g.nz;
        const float p = (float)k - mid;
        zl[s] = p * g.rho;
        zu[s] = (p + 1.0f) * g.rho;
        cl[s] = patch_row_offset(p, cv);
        cup[s] = patch_row_offset(p + 1.0f, cv);
        down[s] = p + 0.5f < 0.0f;
        middle[s] = p + 0.5f == 0.0f;
        pp[s] = down[s] ? p + 1.0f : p;
        pl[s] = pp[s] * g.rho_lo;
    }
    const float zmax = fmaxf(fabsf((float)k0 - mid), fabsf((float)(k0 + 64) - mid)) * g.rho;
    const size_t nuv = (size_t)g.nu * g.nv;
    const unsigned col_bytes = (unsigned)g.nv * 4u;

    float2 sum[4], before[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) sum[q] = before[q] = make_float2(0.0f, 0.0f);

    auto build = [&](int first, int buf) {
#pragma unroll 1
        for (int t = zg; t < PT_ANGLES; t += ZG)
            if (first + t < a_end)
                patch_list(g, wproj, first + t, i0, j0, heads + buf * PT_ANGLES + t,
                           entries + (size_t)(buf * PT_ANGLES + t) * entry_stride, p_edge, edge);
    };
    auto walk = [&](int a, const PatchHead *head, const float4 *ent) {
        const float mag = head->mag;
        const float *pa = wproj + (size_t)a * nuv;
        int rb[2], re[2], r0[2];
        float c0[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const float fb = patch_row(zl[s], mag, cl[s]), fe = patch_row(zu[s], mag, cup[s]);
            rb[s] = __float_as_int(fb);
            re[s] = live[s] ? __float_as_int(fe) : rb[s];
            r0[s] = down[s] ? re[s] - 1 : rb[s];
            c0[s] = ((down[s] ? fe - 1.0f : fb) - ZMAGIC) - cv;
        }
        auto crossing = [&](int s, int t) {            // the t-th row of voxel s
            const int step = down[s] ? -t : t;
            const bool ok = (unsigned)(r0[s] + step - ZMAGIC_BITS) < (unsigned)g.nv && live[s] && !middle[s];
            const float at = patch_crossing(g, c0[s] + (float)step, pp[s], pl[s]);
            return ok ? at : PT_NEVER;
        };
        const int rows = (int)ceilf(__fmaf_rn(g.rho, mag, 1e-3f));
        const bool one = zmax * head->dmag + 2.0f * PT_MARGIN <= 1.0f;
        auto short_rows = [&](auto rows_c) {
            constexpr int ROWS = decltype(rows_c)::value;
            unsigned off[2];
            float2 m[ROWS];
            bool pick[ROWS][2];
            const float2 at[1] = {make_float2(crossing(0, 0), crossing(1, 0))};
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int lo = min(max(down[s] ? re[s] - ROWS : rb[s], ZMAGIC_BITS), ZMAGIC_BITS + g.nv - ROWS);
                off[s] = (unsigned)(lo - ZMAGIC_BITS) * 4u + head->base;
#pragma unroll
                for (int t = 0; t < ROWS; ++t) {
                    const float f = lo + t >= rb[s] && lo + t < re[s] ? 1.0f : 0.0f;
                    if (s == 0) m[t].x = f; else m[t].y = f;
                    pick[t][s] = r0[s] == lo + t;
                }
            }
#pragma unroll
            for (int st = 0; st < PT_MAX_COLUMNS / PT_STEP; ++st) {
                unsigned mask = head->mask[st];
                const float4 *e = ent + st * PT_STEP * 4;
                unsigned o0 = off[0] + st * PT_STEP * col_bytes, o1 = off[1] + st * PT_STEP * col_bytes;
#pragma unroll 2
                for (; mask != 0; mask >>= 4, e += 4, o0 += col_bytes, o1 += col_bytes) {
                    const float *w0 = (const float *)((const char *)pa + (size_t)o0);
                    const float *w1 = (const float *)((const char *)pa + (size_t)o1);
                    float2 w[ROWS];
#pragma unroll
                    for (int t = 0; t < ROWS; ++t) w[t] = make_float2(__ldg(w0 + t), __ldg(w1 + t));
                    float2 S = __fmul2_rn(m[0], w[0]);
                    float2 d[1] = {w[0]};
#pragma unroll
                    for (int t = 1; t < ROWS; ++t) {
                        S = __ffma2_rn(m[t], w[t], S);
                        d[0].x = pick[t][0] ? w[t].x : d[0].x;
                        d[0].y = pick[t][1] ? w[t].y : d[0].y;
                    }
                    patch_cells<1>(mask & 15u, e, S, d, at, sum, before);
                }
            }
        };
        if (one && rows <= 2) {
            short_rows(std::integral_constant<int, 2>());
        } else if (one && rows <= 3) {
            short_rows(std::integral_constant<int, 3>());
        } else {
            // any number of rows; the first two may cross the plane
            const float2 at[2] = {make_float2(crossing(0, 0), crossing(1, 0)),
                                  make_float2(crossing(0, 1), crossing(1, 1))};
            int lo[2], hi[2], dr[2][2];
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                lo[s] = max(rb[s] - ZMAGIC_BITS, 0);
                hi[s] = min(re[s] - ZMAGIC_BITS, g.nv);
#pragma unroll
                for (int t = 0; t < 2; ++t)
                    dr[t][s] = min(max(r0[s] - ZMAGIC_BITS + (down[s] ? -t : t), 0), g.nv - 1);
            }
#pragma unroll 1
            for (int st = 0; st < PT_MAX_COLUMNS / PT_STEP; ++st) {
                unsigned mask = head->mask[st];
                const float4 *e = ent + st * PT_STEP * 4;
                const float *w = (const float *)((const char *)pa + (size_t)(head->base + st * PT_STEP * col_bytes));
#pragma unroll 1
                for (; mask != 0; mask >>= 4, e += 4, w += g.nv) {
                    const float2 d[2] = {make_float2(__ldg(w + dr[0][0]), __ldg(w + dr[0][1])),
                                         make_float2(__ldg(w + dr[1][0]), __ldg(w + dr[1][1]))};
                    float2 S = make_float2(0.0f, 0.0f);
#pragma unroll 4
                    for (int t = 0; t < rows; ++t) {
                        if (lo[0] + t < hi[0]) S.x += __ldg(w + lo[0] + t);
                        if (lo[1] + t < hi[1]) S.y += __ldg(w + lo[1] + t);
                    }
                    patch_cells<2>(mask & 15u, e, S, d, at, sum, before);
                }
            }
        }
    };

    build(a_begin, 0);
    group_sync();
    int buf = 0;
#pragma unroll 1
    for (int a = a_begin; a < a_end; a += PT_ANGLES, buf ^= 1) {
        if (a + PT_ANGLES < a_end) build(a + PT_ANGLES, buf ^ 1);
        const int n = min(PT_ANGLES, a_end - a);
#pragma unroll 1
        for (int t = 0; t < n; ++t)
            walk(a + t, heads + buf * PT_ANGLES + t, entries + (size_t)(buf * PT_ANGLES + t) * entry_stride);
        group_sync();
    }

    // Move the crossing parts: slot k of D goes to voxel k + 1 below the
    // mid-plane and to voxel k - 1 above it; the tile's ends come from `edge`.
    float *const dsh = (float *)mine;                       // [4][SLOTS + 2]
    float *const esh = dsh + 4 * (SLOTS + 2);               // [ZG][8]
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (live[0]) dsh[q * (SLOTS + 2) + 1 + zg * 64 + lane] = before[q].x;
        if (live[1]) dsh[q * (SLOTS + 2) + 33 + zg * 64 + lane] = before[q].y;
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        for (int o = 4; o < 32; o <<= 1) edge[e] += __shfl_xor_sync(0xffffffffu, edge[e], o);
        if (lane < 4) esh[zg * 8 + e * 4 + lane] = edge[e];
    }
    group_sync();
    if (zg == 0 && lane < 8) {
        float s = 0.0f;
        for (int z = 0; z < ZG; ++z) s += esh[z * 8 + lane];
        dsh[(lane & 3) * (SLOTS + 2) + (lane < 4 ? 0 : 1 + kend - kb)] = s;
    }
    group_sync();
    const double acoef = epi_a(epi), bcoef = epi_b(epi);
    double sq = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = i0 + (q & 1), j = j0 + (q >> 1);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int k = k0 + s * 32 + lane;
            if (!live[s] || i >= g.nx || j >= g.ny) continue;
            const float *dk = dsh + q * (SLOTS + 2) + 1 + (k - kb);
            float v = (s == 0 ? sum[q].x : sum[q].y) - dk[0];
            if (2 * k - 1 < g.nz) v += dk[-1];              // slab k - 1 lies below the mid-plane
            if (2 * k + 3 > g.nz) v += dk[1];
            const size_t flat = ((size_t)j * g.nx + i) * g.nz + k;
            if (acc_in) v += acc_in[flat];
            if (acc_out) {
                acc_out[flat] = v;
                continue;
            }
            const size_t o = ZFAST ? (size_t)(zf_col(g, i, j) + k) : ((size_t)k * g.ny + j) * g.nx + i;
            double out = acoef * (double)v;
            if (bcoef != 0.0) {
                const T *oldp = epi.old ? (const T *)epi.old : (const T *)vol;
                out += bcoef * (double)Storage<T>::ld_plain(oldp + o);
            }
            const float stored = Storage<T>::round((float)out);
            Storage<T>::store(vol + o, stored);
            sq += (double)stored * (double)stored;
        }
    }
    double *partial = acc_out ? nullptr : partial_at();
    if (partial) {
        warp_partial(sq, partial);
        if (PATCHES * ZG < TILE_PARTIALS && lane == 0)
            for (int w = PATCHES * ZG + warp; w < TILE_PARTIALS; w += PATCHES * ZG) partial[w] = 0.0;
    }
}

}  // namespace cbct
