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
//   neighbouring slab.  That part is summed apart (D) and moved from voxel to
//   voxel once, after the last angle.  Only a voxel's first row can have one,
//   as long as a plane passes at most one row between the patch's near and far
//   depth (PT_MARGIN included); the general walk takes up to PT_CROSSING.  D
//   is a small part of the sum, so nothing cancels.
//
// A^T y at 256^3 / 512^2 / 360 angles: 37.3 ms with backward_tile, 12.6 here;
// 58 warp instructions per 32 voxels and angle, 63 in the first version
// (169 in backward_tile), issue slots 72 % busy, 71 % of the sectors from L1.
// Relative error against FP64 6.8e-7 -> 5.3e-7: fewer and shorter sums.
// Measured and not kept: prefetching the next column's rows (2.87 against 2.80
// ms per 90 angles) or the next angle's lines (3.48), four voxels per lane
// (3.13), four patches per CTA (2.86).
//
// Geometries outside the bounds of set_patch_bounds (steep cones, voxels that
// cover very many detector columns) take backward_tile.
#pragma once

#include "projector_device.cuh"

namespace cbct {


constexpr int PT_ANGLES = 8;             // angles listed at a time, by all splits of a patch together
constexpr int PT_STEP = 8;               // detector columns listed in one step of a warp (x 4 cells)
constexpr int PT_MAX_COLUMNS = 24;       // PT_BOUND_COLUMNS in steps of PT_STEP
constexpr float PT_MARGIN = 0.05f;       // pixels; covers the windows' rounding (about 1e-4)
constexpr int PT_CROSSING = 3;           // most rows that a plane passes between a patch's near and far depth
constexpr float PT_NEVER = -FLT_MAX;     // crossing alpha of a row that enters its slab before the patch

// Columns of one angle: mask[s] bit 4 c + q: detector column 8 s + c crosses
// cell q; base: byte offset of the first column within the angle's
// projection; mag: magnification at the far depth; dmag: near minus far.
struct PatchHead {
    unsigned mask[PT_MAX_COLUMNS / PT_STEP], base;
    float mag, dmag, pad[2];
};

// Bytes of a list of `angles` angles, two buffers (columns: DevGeom::patch_columns).
__host__ __device__ __forceinline__ int patch_list_bytes(int columns, int angles) {
    return 2 * angles * ((int)sizeof(PatchHead) + columns * 4 * (int)sizeof(float4));
}

// Shared memory of a tile of PATCHES patches, ZG stacks and SPLITS angle ranges: the lists, and
// after the last angle the crossing parts, the edges' sums and the splits' sums.
template <int PATCHES, int ZG, int SPLITS>
__host__ __device__ __forceinline__ int patch_shared_bytes(int columns) {
    const int lists = PATCHES * SPLITS * patch_list_bytes(columns, PT_ANGLES / SPLITS);
    const int last = (int)sizeof(float) * PATCHES * (4 * (64 * ZG + 2) + 8 * ZG * SPLITS + (SPLITS - 1) * ZG * 16 * 32);
    return lists > last ? lists : last;
}

__device__ __forceinline__ float fast_rcp(float v) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
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
// the difference is rounded at its own size only.  p_lo: p rho_lo, plus
// DevGeom::mid_down, which only the middle row (c = 0) on the mid-plane (p = 0)
// feels: with it that row crosses at infinity, so that all of it moves from the
// slab above, where the rows' windows put it, to the slab below; without it the
// crossing is NaN, which saturates to 0.  (A test for the row in the windows
// cost 0.6 to 2.4 % at 256^3, this nothing.)
__device__ __forceinline__ float patch_crossing(const DevGeom &g, float c, float p, float p_lo) {
    const float n = __fmaf_rn(p, g.rho_hi, -(c * g.m_hi)) + __fmaf_rn(-c, g.m_lo, p_lo);
    return n * fast_rcp(c);
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
        const float mag = g.dsd * fast_rcp(g.dso - (px * cs.x + py * cs.y));
        const float u = (py * cs.x - px * cs.y) * mag;
        umin = fminf(umin, u);
        umax = fmaxf(umax, u);
        magmin = fminf(magmin, mag);
        magmax = fmaxf(magmax, mag);
    }
    const float inv_du = fast_rcp(g.du), cu = 0.5f * (g.nu - 1), cv = 0.5f * (g.nv - 1);
    const int iu0 = max(0, (int)ceilf(__fmaf_rn(umin, inv_du, cu - PT_MARGIN)));
    const int iu1 = min(min(g.nu - 1, iu0 + g.patch_columns - 1), (int)floorf(__fmaf_rn(umax, inv_du, cu + PT_MARGIN)));
    const int cell = lane & 3, i = i0 + (cell & 1), j = j0 + (cell >> 1);
    const bool in_volume = i < g.nx && j < g.ny;
    const float dmag = magmax - magmin;
#pragma unroll 1
    for (int s = 0; s < PT_MAX_COLUMNS / PT_STEP; ++s) {
        if (lane == 0) head->mask[s] = 0;
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
        const unsigned crossed = __ballot_sync(0xffffffffu, crosses);
        if (lane == 0) head->mask[s] = crossed;
        if (crosses) {
            const float len = aout - ain, inv = fast_rcp(len), start = -ain * inv;
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
                const int n = (int)ceilf(__fmaf_rn(fabsf(rows), dmag, 2.0f * PT_MARGIN));
                for (int t = 0; t < n; ++t, row += step) {
                    if ((unsigned)row >= (unsigned)g.nv) continue;
                    const float at = patch_crossing(g, (float)row - cv, p, p * g.rho_lo);
                    edge[e] = __fmaf_rn(fma_sat(at, inv, start), len * __ldg(wcol + row), edge[e]);
                }
            }
        }
    }
    if (lane == 0) {
        head->base = (unsigned)iu0 * (unsigned)g.nv * 4u;
        head->mag = magmin;
        head->dmag = dmag;
    }
}

// Adds one detector column's part to the cells it crosses (bits of `cells`),
// for the lane's two voxels.  S: the sum of each voxel's rows; d[t]: its t-th
// row from the entry plane, at[t]: the alpha at which that row enters the
// voxel's slab.
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

__device__ __forceinline__ float &half(float2 &v, int s) { return s ? v.y : v.x; }

// A tile: PATCHES patches of 2 x 2 columns side by side (along x if ALONG_X,
// else along y), ZG stacks of 64 voxels, and the angles in SPLITS ranges, 8
// warps in all.  The splits' sums are added in order at the end; they keep the
// GPU busy with a volume that is not deep (32^3 voxels are 256 patches).
// Angles [a_begin, a_end), running sums and epilogue as in backward_tile.
// lists: patch_shared_bytes<PATCHES, ZG, SPLITS>() of shared memory.
template <typename T, bool ZFAST, int PATCHES, bool ALONG_X, int ZG, int SPLITS, typename PartialAt>
__device__ __forceinline__ void patch_tile(const DevGeom &g, const float *__restrict__ wproj, T *__restrict__ vol,
                                           const Epilogue &epi, int tx, int ty, int tz, int a_begin, int a_end,
                                           const float *acc_in, float *acc_out, PartialAt &&partial_at, char *lists) {
    static_assert(PATCHES * ZG * SPLITS == TILE_PARTIALS, "one norm partial per warp");
    constexpr int DEPTH = 64, SLOTS = DEPTH * ZG, ANGLES = PT_ANGLES / SPLITS;
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const int zg = warp % ZG, patch = warp / ZG % PATCHES, split = warp / (ZG * PATCHES);
    const int i0 = tx * (ALONG_X ? 2 * PATCHES : 2) + (ALONG_X ? 2 * patch : 0);
    const int j0 = ty * (ALONG_X ? 2 : 2 * PATCHES) + (ALONG_X ? 0 : 2 * patch);
    const int kb = tz * SLOTS, k0 = kb + zg * DEPTH;
    const int kend = min(kb + SLOTS, g.nz);
    const int angles = a_end - a_begin, group = split * PATCHES + patch;
    const int a_first = a_begin + (int)((long long)angles * split / SPLITS);
    const int a_last = a_begin + (int)((long long)angles * (split + 1) / SPLITS);
    const float cv = 0.5f * (g.nv - 1), mid = 0.5f * g.nz;
    auto group_sync = [&]() {               // the warps that share a list
        if (ZG == 1)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(32 * ZG) : "memory");
    };
    char *const mine = lists + group * patch_list_bytes(g.patch_columns, ANGLES);
    const int entry_stride = g.patch_columns * 4;
    PatchHead *const heads = (PatchHead *)mine;
    float4 *const entries = (float4 *)(mine + 2 * ANGLES * sizeof(PatchHead));

    // planes at the ends of the tile's slabs, when rays cross them outwards
    // (or the middle row moves down across the tile's end)
    const float p_edge[2] = {fminf((float)kb - mid, 0.0f), fmaxf((float)kend - mid, (float)kend == mid ? g.mid_down : 0.0f)};
    float edge[2] = {0.0f, 0.0f};

    const float pk = (float)(k0 + lane) - mid;          // lower plane of the lane's first voxel, from the mid-plane
    // every ray of the warp goes down (-1) / up (1), or not (0: the slabs around the mid-plane)
    const int direction = (float)(k0 + DEPTH) - mid <= 0.0f ? -1 : (float)k0 - mid >= 0.0f ? 1 : 0;
    const float zmax = fmaxf(fabsf((float)k0 - mid), fabsf((float)(k0 + DEPTH) - mid)) * g.rho;
    const size_t nuv = (size_t)g.nu * g.nv;
    const int segments = (g.patch_columns + PT_STEP - 1) / PT_STEP;
    const unsigned col_bytes = (unsigned)g.nv * 4u;

    float2 sum[4], before[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) sum[q] = before[q] = make_float2(0.0f, 0.0f);

    auto build = [&](int first, int buf) {
#pragma unroll 1
        for (int t = zg; t < ANGLES; t += ZG)
            if (first + t < a_last)
                patch_list(g, wproj, first + t, i0, j0, heads + buf * ANGLES + t,
                           entries + (size_t)(buf * ANGLES + t) * entry_stride, p_edge, edge);
    };
    // Calls column(bits of the crossed cells, entries, byte offset) for every detector column of an angle.
    auto columns = [&](const PatchHead *head, const float4 *ent, auto &&column) {
#pragma unroll 1
        for (int st = 0; st < segments; ++st) {
            unsigned mask = head->mask[st];
            unsigned col = st * PT_STEP * col_bytes;
            const float4 *e = ent + st * PT_STEP * 4;
#pragma unroll 1
            for (; mask != 0; mask >>= 4, e += 4, col += col_bytes) column(mask & 15u, e, col);
        }
    };
    // Voxels of at most ROWS rows, one of which may cross the entry plane.  A
    // voxel's rows are [fb, fe) (plus ZMAGIC); the loads cover ROWS rows from
    // `lo`, weighted m (1: the voxel's).  DIR +-1: all rows of the warp lie on
    // the detector and all rays go one way, so that lo = fb or fe - ROWS, and
    // the row that may cross is the first or the last one loaded; otherwise
    // (0) that row has weight f.  Scalar arithmetic: the packed forms take no
    // constant operands.
    auto short_rows = [&](const float *pa, const PatchHead *head, const float4 *ent, auto rows_c, auto dir_c) {
        constexpr int ROWS = decltype(rows_c)::value, DIR = decltype(dir_c)::value;
        const float mag = head->mag;
        float2 m[ROWS], f[DIR == 0 ? ROWS : 1], at[1];
        unsigned o[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const float p = pk + 32.0f * s;
            float fb = patch_row(p * g.rho, mag, DIR > 0 ? cv - PT_MARGIN : DIR < 0 ? cv + PT_MARGIN : patch_row_offset(p, cv));
            float fe = patch_row((p + 1.0f) * g.rho, mag, DIR > 0 ? cv - PT_MARGIN : patch_row_offset(p + 1.0f, cv));
            const bool down = DIR < 0 || (DIR == 0 && p < -0.5f);
            const float pe = down ? p + 1.0f : p;
            const float first = down ? fe - 1.0f : fb;
            const float c = (first - ZMAGIC) - cv;
            float a = patch_crossing(g, c, pe, __fmaf_rn(pe, g.rho_lo, g.mid_down));
            float lo = down ? fe - (float)ROWS : fb;
            if (DIR == 0) {
                lo = fminf(fmaxf(lo, ZMAGIC), ZMAGIC + (float)(g.nv - ROWS));
                if (p == -0.5f) a = PT_NEVER;               // the slab around the mid-plane: no ray enters it
                if (k0 + s * 32 + lane >= g.nz) fe = fb;
                fe = fminf(fe, ZMAGIC + (float)g.nv);
                fb = fmaxf(fb, ZMAGIC);
            }
            half(at[0], s) = a;
            o[s] = (unsigned)__float_as_int(lo) * 4u + (head->base - (unsigned)ZMAGIC_BITS * 4u);
#pragma unroll
            for (int t = 0; t < ROWS; ++t) {
                float w;
                if (DIR > 0)
                    w = __saturatef((fe - fb) - (float)t);
                else if (DIR < 0)
                    w = __saturatef((fe - fb) - (float)(ROWS - 1 - t));
                else {
                    w = __saturatef((fe - lo) - (float)t) - __saturatef((fb - lo) - (float)t);
                    half(f[t], s) = __saturatef(1.0f - fabsf((first - lo) - (float)t));
                }
                half(m[t], s) = w;
            }
        }
        columns(head, ent, [&](unsigned cells, const float4 *e, unsigned col) {
            const float *w0 = (const float *)((const char *)pa + (size_t)(o[0] + col));
            const float *w1 = (const float *)((const char *)pa + (size_t)(o[1] + col));
            float2 w[ROWS];
#pragma unroll
            for (int t = 0; t < ROWS; ++t) w[t] = make_float2(__ldg(w0 + t), __ldg(w1 + t));
            float2 S = __fmul2_rn(m[0], w[0]), d[1];
#pragma unroll
            for (int t = 1; t < ROWS; ++t) S = __ffma2_rn(m[t], w[t], S);
            if (DIR != 0) {
                d[0] = w[DIR > 0 ? 0 : ROWS - 1];
            } else {
                d[0] = __fmul2_rn(f[0], w[0]);
#pragma unroll
                for (int t = 1; t < ROWS; ++t) d[0] = __ffma2_rn(f[DIR == 0 ? t : 0], w[t], d[0]);
            }
            patch_cells<1>(cells, e, S, d, at, sum, before);
        });
    };
    auto walk = [&](const float *pa, const PatchHead *head, const float4 *ent) {
        const float mag = head->mag;
        const float most = __fmaf_rn(g.rho, mag, 1e-3f);
        const bool one = zmax * head->dmag + 2.0f * PT_MARGIN <= 1.0f;
        typedef std::integral_constant<int, 0> C0;
        typedef std::integral_constant<int, 1> C1;
        typedef std::integral_constant<int, -1> CM;
        typedef std::integral_constant<int, 2> C2;
        typedef std::integral_constant<int, 3> C3;
        if (one && most <= 3.0f) {
            if (direction == 0 || __fmaf_rn(zmax, mag, 5.0f) > cv)
                short_rows(pa, head, ent, C3(), C0());
            else if (direction > 0)
                most <= 2.0f ? short_rows(pa, head, ent, C2(), C1()) : short_rows(pa, head, ent, C3(), C1());
            else
                most <= 2.0f ? short_rows(pa, head, ent, C2(), CM()) : short_rows(pa, head, ent, C3(), CM());
            return;
        }
        // any number of rows; up to PT_CROSSING of them may cross the plane
        const int crossing_rows = (int)ceilf(__fmaf_rn(zmax, head->dmag, 2.0f * PT_MARGIN));
        const int rows = (int)ceilf(most);
        float2 at[PT_CROSSING];
        int lo[2], hi[2], first[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const float p = pk + 32.0f * s;
            const float fb = patch_row(p * g.rho, mag, patch_row_offset(p, cv));
            const float fe = patch_row((p + 1.0f) * g.rho, mag, patch_row_offset(p + 1.0f, cv));
            const bool down = p < -0.5f, live = k0 + s * 32 + lane < g.nz;
            const float pe = down ? p + 1.0f : p;
            const float c = ((down ? fe - 1.0f : fb) - ZMAGIC) - cv;
            const int rb = __float_as_int(fb) - ZMAGIC_BITS, re = __float_as_int(fe) - ZMAGIC_BITS;
            lo[s] = max(rb, 0);
            hi[s] = live ? min(re, g.nv) : lo[s];
            first[s] = down ? re - 1 : rb;
#pragma unroll
            for (int t = 0; t < PT_CROSSING; ++t) {
                const int step = down ? -t : t;
                const bool ok = t < crossing_rows && live && p != -0.5f && (unsigned)(first[s] + step) < (unsigned)g.nv;
                half(at[t], s) = ok ? patch_crossing(g, c + (float)step, pe, __fmaf_rn(pe, g.rho_lo, g.mid_down)) : PT_NEVER;
            }
        }
        // on the detector and all one way: every voxel has the first `full`
        // rows, and the rows that may cross need no clamp
        const bool inside = direction != 0 && __fmaf_rn(zmax, mag, most + (float)(PT_CROSSING + 2)) <= cv;
        const int full = inside ? (int)(most - (PT_MARGIN + 2e-3f)) : 0;
        const unsigned base = head->base;
        columns(head, ent, [&](unsigned cells, const float4 *e, unsigned col) {
            const float *w = (const float *)((const char *)pa + (size_t)(base + col));
            float2 S = make_float2(0.0f, 0.0f), d[PT_CROSSING];
            const float *w0 = w + lo[0], *w1 = w + lo[1];
#pragma unroll 2
            for (int t = 0; t < full; ++t) S = __fadd2_rn(S, make_float2(__ldg(w0 + t), __ldg(w1 + t)));
#pragma unroll 1
            for (int t = full; t < rows; ++t) {
                if (lo[0] + t < hi[0]) S.x += __ldg(w0 + t);
                if (lo[1] + t < hi[1]) S.y += __ldg(w1 + t);
            }
            if (inside) {
                const float *f0 = w + first[0], *f1 = w + first[1];
#pragma unroll
                for (int t = 0; t < PT_CROSSING; ++t, f0 += direction, f1 += direction)
                    d[t] = t < crossing_rows ? make_float2(__ldg(f0), __ldg(f1)) : make_float2(0.0f, 0.0f);
            } else {
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const int step = pk + 32.0f * s < -0.5f ? -1 : 1;
#pragma unroll
                    for (int t = 0; t < PT_CROSSING; ++t)
                        half(d[t], s) = t < crossing_rows ? __ldg(w + min(max(first[s] + t * step, 0), g.nv - 1)) : 0.0f;
                }
            }
            if (crossing_rows <= 1) {
                const float2 d1[1] = {d[0]}, at1[1] = {at[0]};
                patch_cells<1>(cells, e, S, d1, at1, sum, before);
            } else {
                patch_cells<PT_CROSSING>(cells, e, S, d, at, sum, before);
            }
        });
    };

    build(a_first, 0);
    group_sync();
    int buf = 0;
    const float *pa = wproj + (size_t)a_first * nuv;
#pragma unroll 1
    for (int a = a_first; a < a_last; a += ANGLES, buf ^= 1) {
        if (a + ANGLES < a_last) build(a + ANGLES, buf ^ 1);
        if (k0 < g.nz) {                    // a warp past the volume only helps with the lists
            const int n = min(ANGLES, a_last - a);
            const PatchHead *head = heads + buf * ANGLES;
            const float4 *ent = entries + (size_t)(buf * ANGLES) * entry_stride;
#pragma unroll 1
            for (int t = 0; t < n; ++t, ++head, ent += entry_stride, pa += nuv) walk(pa, head, ent);
        }
        group_sync();
    }

    // Add the splits' sums, in order, to the first split's.
    float *const dsh = (float *)lists + patch * 4 * (SLOTS + 2);                        // [patch][4][SLOTS + 2]
    float *const esh = (float *)lists + PATCHES * 4 * (SLOTS + 2) + patch * 8 * ZG * SPLITS;
    float *const rsh = (float *)lists + PATCHES * (4 * (SLOTS + 2) + 8 * ZG * SPLITS);
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        for (int o = 4; o < 32; o <<= 1) edge[e] += __shfl_xor_sync(0xffffffffu, edge[e], o);
        if (lane < 4) esh[(split * ZG + zg) * 8 + e * 4 + lane] = edge[e];
    }
    if (SPLITS > 1) {
        float *const own = rsh + ((patch * ZG + zg) * 16) * 32 + lane;
        constexpr int STRIDE = PATCHES * ZG * 16 * 32;
        if (split > 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float *const to = own + (split - 1) * STRIDE + q * 4 * 32;
                to[0] = sum[q].x;
                to[32] = sum[q].y;
                to[64] = before[q].x;
                to[96] = before[q].y;
            }
        }
        __syncthreads();
        if (split == 0) {
#pragma unroll 1
            for (int o = 0; o < SPLITS - 1; ++o) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float *const from = own + o * STRIDE + q * 4 * 32;
                    sum[q].x += from[0];
                    sum[q].y += from[32];
                    before[q].x += from[64];
                    before[q].y += from[96];
                }
            }
        }
    }

    // Move the crossing parts: slot k of D goes to voxel k + 1 below the
    // mid-plane and to voxel k - 1 above it; the tile's ends come from `edge`.
    if (split == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
            for (int s = 0; s < 2; ++s)
                if (k0 + s * 32 + lane < g.nz) dsh[q * (SLOTS + 2) + 1 + zg * DEPTH + s * 32 + lane] = half(before[q], s);
        }
    }
    __syncthreads();
    if (split == 0 && zg == 0 && lane < 8) {
        float v = 0.0f;
        for (int w = 0; w < ZG * SPLITS; ++w) v += esh[w * 8 + lane];
        dsh[(lane & 3) * (SLOTS + 2) + (lane < 4 ? 0 : 1 + kend - kb)] = v;
    }
    __syncthreads();
    const double acoef = epi_a(epi), bcoef = epi_b(epi);
    double sq = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = i0 + (q & 1), j = j0 + (q >> 1);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int k = k0 + s * 32 + lane;
            if (split > 0 || k >= g.nz || i >= g.nx || j >= g.ny) continue;
            const float *dk = dsh + q * (SLOTS + 2) + 1 + (k - kb);
            float v = half(sum[q], s) - dk[0];
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
    if (partial) warp_partial(sq, partial);
}

}  // namespace cbct
