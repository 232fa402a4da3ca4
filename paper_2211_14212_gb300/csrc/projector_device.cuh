// Device-side building blocks of the cone-beam projectors (Sec. 1, Eq. 1):
// the ray traversal shared by A and A^T, and one tile of each projector,
// callable from a plain grid (projector.cu) or from a persistent kernel that
// walks a work list spanning several problems (serve.cu).
//
// Work layout ("ray-column warps").  In a circular cone-beam scan every ray of
// one detector column (angle a, column iu) has the same projection onto the
// xy plane, so all of them cross the x and y voxel planes at the same alpha
// (the x/y tables depend on (a, iu) only).  A warp therefore takes rays of one
// detector column: lane l follows rows iv0 + r * 32 + l for r = 0..R-1.  The
// sequence of x/y cells is the same in all lanes and is computed once for the
// warp's 32 R rays; each ray only tracks its own z crossings, which are rare
// (|dz/d| <= the cone half-angle).  Volumes are read in a z-fastest layout
// x[j][i][k] so that the lanes of one row group, which sit at ~17 consecutive
// k of one voxel column, gather one contiguous run.
//
// Both projectors take every x/y plane crossing from the per-ray tables of
// DevGeom through plane_alpha, and their z crossings from equivalent forms, so
// the backprojector is the transpose of the forward projector, not an
// approximation of it (the paper traces Krylov instabilities to unmatched
// backprojectors, Sec. 2.1.4 and Sec. 4); in FP32 their segment lengths agree
// to rounding.
#pragma once

#include <cfloat>
#include <type_traits>

#include "common.cuh"

namespace cbct {

// One axis of one ray: offset f = plane(pq) - q, inverse direction I, and the
// index pq of the plane nearest to the ray origin (the fixed voxel index when
// I == 0, a ray parallel to the axis' planes).
struct RayAxis {
    float f, I, pq;
};

// Alpha at which a ray crosses plane pq + r of one axis (plane spacing delta):
// (r * delta + f) * I, rounded twice.  Both projectors use only this.
__device__ __forceinline__ float plane_alpha(float r, float delta, const RayAxis &a) {
    return __fmul_rn(__fmaf_rn(r, delta, a.f), a.I);
}

// One axis of the traversal: current voxel index i, step s (+1/-1, 0 when the
// ray is parallel to the axis' planes), index of the plane through which the
// ray leaves the current voxel (relative to pq, as float) and the alpha of
// that crossing.
struct Axis {
    int i, s;
    float r, e;
};

// Clip alpha interval [amin, amax] to the slab between planes plo and phi.
__device__ __forceinline__ void clip_slab(const RayAxis &ra, float delta, int plo, int phi, float &amin,
                                          float &amax, bool &miss) {
    if (ra.I == 0.0f) {
        if (!(ra.pq >= (float)plo && ra.pq < (float)phi)) miss = true;
        return;
    }
    const float a0 = plane_alpha((float)plo - ra.pq, delta, ra), a1 = plane_alpha((float)phi - ra.pq, delta, ra);
    amin = fmaxf(amin, fminf(a0, a1));
    amax = fminf(amax, fmaxf(a0, a1));
}

// Voxel index on one axis at alpha0, within [lo - 1, hi] (lo - 1 and hi stand
// for "before" and "beyond" the range).  The estimate from the ray position is
// corrected by comparing with the crossing alphas themselves, so the result is
// exactly the voxel whose alpha interval [entry, exit) contains alpha0.  The
// exit crossing is returned; it is FLT_MAX when the ray is outside the range
// and moving away from it.
__device__ __forceinline__ Axis axis_start(const RayAxis &ra, float delta, float alpha0, int lo, int hi) {
    Axis st;
    if (ra.I == 0.0f) {         // parallel: fixed index, never crossed
        st.i = (int)ra.pq;
        st.s = 0;
        st.r = 0.0f;
        st.e = FLT_MAX;
        return st;
    }
    // plane coordinate of the ray at alpha0: pq + (alpha0 / I - f) / delta
    int i = (int)floorf(ra.pq + (__fdividef(alpha0, ra.I) - ra.f) / delta);
    i = max(lo - 1, min(hi, i));
    auto al = [&](int p) { return plane_alpha((float)p - ra.pq, delta, ra); };
    if (ra.I > 0.0f) {          // alpha grows with the plane index: voxel i = [alpha(i), alpha(i+1))
        if (i < hi && al(i + 1) <= alpha0) ++i;
        if (i >= lo && al(i) > alpha0) --i;
        st.s = 1;
        st.r = (float)(i + 1) - ra.pq;
        st.e = i < hi ? plane_alpha(st.r, delta, ra) : FLT_MAX;
    } else {                    // alpha falls with the plane index: voxel i = [alpha(i+1), alpha(i))
        if (i >= lo && al(i) <= alpha0) --i;
        if (i < hi && al(i + 1) > alpha0) ++i;
        st.s = -1;
        st.r = (float)i - ra.pq;
        st.e = i >= lo ? plane_alpha(st.r, delta, ra) : FLT_MAX;
    }
    st.i = i;
    return st;
}

// Walk R rays of one detector column (shared xy tables rx, ry; z tables
// rz[r]) through the box [lox,hix) x [loy,hiy) x [loz,hiz) of voxels.  For
// every segment inside the box it calls
//     add(r, alpha_length, value),   value = fetch(cell + k),
//     cell = off + i * sx + j * sy,
// in order along each ray (cell is kept incrementally, so the caller picks the
// linear layout through off, sx, sy).  The value of the voxel a ray occupies
// when it enters the next xy cell is fetched before the current cell's
// segments are added, so each lane keeps R loads in flight across the
// latency of a step; a z crossing inside a cell (rare) fetches the new voxel
// on the spot.  Segments of rays outside [loz, hiz) are added with length 0
// and no fetch.  Returns false (uniformly across the warp) if the xy
// projection misses the box.
template <int R, typename Fetch, typename Add>
__device__ __forceinline__ bool trace_columns(const DevGeom &g, const RayAxis &rx, const RayAxis &ry,
                                              const RayAxis (&rz)[R], int lox, int hix, int loy, int hiy,
                                              int loz, int hiz, int off, int sx, int sy, Fetch &&fetch,
                                              Add &&add) {
    float amin = -FLT_MAX, amax = FLT_MAX;
    bool miss = false;
    clip_slab(rx, g.dx, lox, hix, amin, amax, miss);
    clip_slab(ry, g.dy, loy, hiy, amin, amax, miss);
    if (miss || !(amin < amax)) return false;

    Axis ax = axis_start(rx, g.dx, amin, lox, hix);
    Axis ay = axis_start(ry, g.dy, amin, loy, hiy);
    Axis az[R];
    bool inz[R];
    float cur[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        az[r] = axis_start(rz[r], g.dz, amin, loz, hiz);
        if (az[r].s == 0 && (az[r].i < loz || az[r].i >= hiz)) az[r].i = loz - 1;   // parallel outside
        inz[r] = az[r].i >= loz && az[r].i < hiz;
        cur[r] = amin;
    }
    int cell = off + ax.i * sx + ay.i * sy;
    const int dcx = ax.s * sx, dcy = ay.s * sy;
    float vnext[R];
#pragma unroll
    for (int r = 0; r < R; ++r) vnext[r] = inz[r] ? fetch(cell + az[r].i) : 0.0f;
    const int maxsteps = (hix - lox) + (hiy - loy) + 1;
#pragma unroll 1
    for (int n = 0; n < maxsteps; ++n) {
        const float e = fminf(ax.e, ay.e);
        float v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = vnext[r];
        float zmin = az[0].e;
#pragma unroll
        for (int r = 1; r < R; ++r) zmin = fminf(zmin, az[r].e);
        if (zmin < e) {                    // some ray of this lane crosses a z plane in this xy cell
#pragma unroll
            for (int r = 0; r < R; ++r) {
#pragma unroll 1
                while (az[r].e < e) {
                    if (inz[r]) add(r, az[r].e - cur[r], v[r]);
                    cur[r] = az[r].e;
                    az[r].i += az[r].s;
                    az[r].r += (float)az[r].s;
                    inz[r] = az[r].i >= loz && az[r].i < hiz;
                    az[r].e = inz[r] ? plane_alpha(az[r].r, g.dz, rz[r]) : FLT_MAX;
                    v[r] = inz[r] ? fetch(cell + az[r].i) : 0.0f;
                }
            }
        }
        float len[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            len[r] = inz[r] ? e - cur[r] : 0.0f;
            cur[r] = e;
        }
        bool done;
        if (e == ax.e) {
            ax.i += ax.s;
            done = (unsigned)(ax.i - lox) >= (unsigned)(hix - lox);
            if (!done) {
                cell += dcx;
                ax.r += (float)ax.s;
                ax.e = plane_alpha(ax.r, g.dx, rx);
            }
        } else {
            ay.i += ay.s;
            done = (unsigned)(ay.i - loy) >= (unsigned)(hiy - loy);
            if (!done) {
                cell += dcy;
                ay.r += (float)ay.s;
                ay.e = plane_alpha(ay.r, g.dy, ry);
            }
        }
        if (!done) {
#pragma unroll
            for (int r = 0; r < R; ++r) vnext[r] = inz[r] ? fetch(cell + az[r].i) : 0.0f;
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (inz[r]) add(r, len[r], v[r]);
        if (done) break;
    }
    return true;
}

// xy tables of column (a, iu) and z tables of R rows iv0 + r * 32 + lane; rows
// outside [0, nv) (or past `row_end`) get a z axis that is parallel and
// outside every box, so the lane follows the warp without effect.
template <int R>
__device__ __forceinline__ void load_rays(const DevGeom &g, int a, int iu, int iv0, int row_end, RayAxis &rx,
                                          RayAxis &ry, RayAxis (&rz)[R]) {
    const float4 xy = g.ray_xy[(size_t)a * g.nu + iu];
    const float2 q = g.ray_xyq[(size_t)a * g.nu + iu];
    rx = RayAxis{xy.x, xy.y, q.x};
    ry = RayAxis{xy.z, xy.w, q.y};
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int iv = iv0 + r * 32 + lane;
        if (iv < row_end) {
            const float4 z = g.ray_z[iv];
            rz[r] = RayAxis{z.x, z.y, z.z};
        } else {
            rz[r] = RayAxis{0.0f, 0.0f, (float)(g.nz + 1)};
        }
    }
}

// ------------------------------------------------ x/y cells of a column
//
// All rays of one detector column cross the x and y planes at the same alphas,
// so the sequence of x/y cells a warp walks is the same in its 32 lanes.  The
// lanes compute it together, CELL_CHUNK = 32 crossings at a time: lane l takes
// the l-th next x plane and the l-th next y plane, finds how many crossings of
// the other axis come before each (an estimate from the plane spacing, put
// right by comparing plane_alpha values), and writes its crossings at their
// ranks of the merged sequence.  An entry of the list is the alpha at which a
// cell ends and the linear index of the cell's voxel column.  Stepping the two
// axes in every lane instead took about 40 of the 95 instructions the warp
// spent per cell; the list takes 3 per cell.
constexpr int CELL_CHUNK = 32;

struct CellList {
    RayAxis rx, ry;
    float rxn, ryn;          // next plane of each axis, relative to pq
    float sx, sy;            // +1 / -1, 0 when the column is parallel to the axis' planes
    float ix, iy;            // planes per alpha (0 when parallel)
    unsigned col;            // voxel column of the current cell (zf_col)
    unsigned dcx, dcy;       // its change across an x / y plane
    unsigned colmax;         // largest column index
    float amax;
};

// Sets the list up for the box [0, nx) x [0, ny); false (warp-uniform) if the
// column misses it.  *amin: alpha at which the column enters.
__device__ __forceinline__ bool cells_begin(const DevGeom &g, const RayAxis &rx, const RayAxis &ry, CellList &c,
                                            float *amin) {
    float lo = -FLT_MAX, hi = FLT_MAX;
    bool miss = false;
    clip_slab(rx, g.dx, 0, g.nx, lo, hi, miss);
    clip_slab(ry, g.dy, 0, g.ny, lo, hi, miss);
    if (miss || !(lo < hi)) return false;
    const Axis ax = axis_start(rx, g.dx, lo, 0, g.nx);
    const Axis ay = axis_start(ry, g.dy, lo, 0, g.ny);
    c.rx = rx;
    c.ry = ry;
    c.rxn = ax.r;
    c.ryn = ay.r;
    c.sx = (float)ax.s;
    c.sy = (float)ay.s;
    c.ix = ax.s ? 1.0f / fabsf(g.dx * rx.I) : 0.0f;
    c.iy = ay.s ? 1.0f / fabsf(g.dy * ry.I) : 0.0f;
    c.col = (unsigned)zf_col(g, ax.i, ay.i);
    c.dcx = (unsigned)(ax.s * (g.nz + 2));
    c.dcy = (unsigned)(ay.s * g.nx * (g.nz + 2));
    c.colmax = (unsigned)zf_col(g, g.nx - 1, g.ny - 1);
    c.amax = hi;
    *amin = lo;
    return true;
}

// Writes the next cells (at most CELL_CHUNK) to `list`, padded with empty
// cells to CELL_CHUNK, and returns their number; *last is set when the last
// one ends at amax.  `bias` is added to every column index.  All lanes call
// it; the values of an earlier chunk must not be in use any more.
// The estimates of a crossing's rank are right to one: both axes' alphas carry
// a relative rounding error of a few 2^-24 and the planes of an axis are at
// least 1 / n of their largest alpha apart.  Column indices are clamped to the
// volume, so that no rounding can send a load out of it.
__device__ __forceinline__ int cells_next(const DevGeom &g, CellList &c, unsigned bias, float2 *list, bool *last) {
    const int lane = threadIdx.x & 31;
    constexpr float most = (float)CELL_CHUNK;
    auto alx = [&](float m) { return c.sx != 0.0f ? plane_alpha(__fmaf_rn(c.sx, m, c.rxn), g.dx, c.rx) : FLT_MAX; };
    auto aly = [&](float m) { return c.sy != 0.0f ? plane_alpha(__fmaf_rn(c.sy, m, c.ryn), g.dy, c.ry) : FLT_MAX; };
    const float lf = (float)lane;
    const float ex = alx(lf), ey = aly(lf);
    const float ex0 = __shfl_sync(0xffffffffu, ex, 0), ey0 = __shfl_sync(0xffffffffu, ey, 0);
    // y crossings before ex (strictly), x crossings up to ey: an x crossing
    // comes first where both coincide
    float ny = fminf(fmaxf(ceilf((ex - ey0) * c.iy), 0.0f), most);
    const bool ny_high = ny > 0.0f && aly(ny - 1.0f) >= ex, ny_low = aly(ny) < ex;
    ny = ny_high ? ny - 1.0f : ny_low ? ny + 1.0f : ny;
    float nx = fminf(fmaxf(floorf((ey - ex0) * c.ix) + 1.0f, 0.0f), most);
    const bool nx_high = nx > 0.0f && alx(nx - 1.0f) > ey, nx_low = alx(nx) <= ey;
    nx = nx_high ? nx - 1.0f : nx_low ? nx + 1.0f : nx;
    const int nxi = (int)nx, nyi = (int)ny;
    const int rank_x = lane + nyi, rank_y = lane + nxi;
    const unsigned cx = min(c.col + (unsigned)lane * c.dcx + (unsigned)nyi * c.dcy, c.colmax) + bias;
    const unsigned cy = min(c.col + (unsigned)nxi * c.dcx + (unsigned)lane * c.dcy, c.colmax) + bias;
    __syncwarp();
    if (rank_x < CELL_CHUNK) list[rank_x] = make_float2(ex, __uint_as_float(cx));
    if (rank_y < CELL_CHUNK) list[rank_y] = make_float2(ey, __uint_as_float(cy));
    const int used_x = __popc(__ballot_sync(0xffffffffu, rank_x < CELL_CHUNK));
    __syncwarp();
    const float2 own = list[lane];
    const int inside = __popc(__ballot_sync(0xffffffffu, own.x < c.amax));
    const int n = min(inside + 1, CELL_CHUNK);
    const float tail = __shfl_sync(0xffffffffu, own.y, n - 1);
    list[lane] = make_float2(fminf(own.x, c.amax), lane < n ? own.y : tail);
    __syncwarp();
    c.rxn += c.sx * (float)used_x;
    c.ryn += c.sy * (float)(CELL_CHUNK - used_x);
    c.col += (unsigned)used_x * c.dcx + (unsigned)(CELL_CHUNK - used_x) * c.dcy;
    *last = inside < CELL_CHUNK;
    return n;
}

// ------------------------------------------- z index from alpha (forward)
//
// Along a ray the z voxel coordinate is linear in alpha.  Measured from the
// plane pq nearest to the ray origin, in the direction in which the ray leaves
// the mid-plane (upwards for v > 0, downwards for v < 0: the source is at
// z = 0, so every ray only moves away from it), it is t = a * alpha + b with
// a >= 0.  The next plane ceil(t) comes from one add rounded up: t + m, with
// m = 1.5 * 2^23 + c, leaves an integer whose float bits are one more than the
// voxel index (up: c = pq) or than its mirror image (down: c = -pq), plus a
// constant that is folded into the column's address.  The part of a cell (in
// voxel units of z) that lies past that plane is sat(t_exit - ceil(t_entry)).
// t is clamped to less than one voxel past the volume's end, where the padded
// columns hold zeros.
constexpr float ZMAGIC = 12582912.0f;        // 1.5 * 2^23
constexpr int ZMAGIC_BITS = 0x4B400000;

struct RayZ {
    float a, b;          // t = a * alpha + b (voxel units)
    float inva;          // alpha per voxel (0: parallel to the z planes)
    float m;             // ZMAGIC + c
    float hi;            // clamp of t
    bool down;
};
constexpr float ZPAST = 0.99609375f;         // how far past the volume's end t may go

// `down` is the direction to use for a ray without one of its own.
__device__ __forceinline__ RayZ make_rayz(const RayAxis &rz, float dz, int nz, bool down) {
    RayZ r;
    if (rz.I == 0.0f) {                          // parallel to the z planes: fixed voxel (pads: outside)
        const float k = fminf(rz.pq, (float)nz);
        r.a = r.inva = 0.0f;
        r.b = 0.5f;
        r.down = down;
        r.m = ZMAGIC + (down ? -1.0f - k : k);
        r.hi = 0.5f + ZPAST;
    } else {
        r.down = rz.I < 0.0f;
        r.inva = fabsf(dz * rz.I);
        r.a = 1.0f / r.inva;
        const float b = rz.f / dz;
        r.b = r.down ? b : -b;
        r.m = ZMAGIC + (r.down ? -rz.pq : rz.pq);
        r.hi = (r.down ? rz.pq : (float)nz - rz.pq) + ZPAST;
    }
    return r;
}

// Walks R rays of one detector column through the padded z-fastest volume, for
// geometries with at most one z-plane crossing per xy cell
// (DevGeom::zsingle).  In every cell of alpha length L a ray adds
//     L v + (part past the next plane) (vn - v),
// v and vn the voxel it entered the cell in and its neighbour across that
// plane: both are loaded for every cell (one address, the neighbour at a fixed
// offset), so no lane branches.  DIR: +1 / -1 when every ray of the warp goes
// up / down, 0 when both occur (the row group around the mid-plane); CLAMP:
// some ray leaves the volume through its top or bottom.  OFF32: the padded volume
// has at most 2^32 bytes (OFF32_BYTES), so a voxel's address is one 32-bit
// multiply-add from the volume's base instead of a 64-bit one.  Ray pairs use packed
// FP32x2 arithmetic.  The sums of a chunk of cells are folded into acc every
// CELL_CHUNK cells; for 16-bit storage (COMP) every cell's term is added to
// acc with Kahan compensation (FP16 at 256^3 / 512^2 / 360 angles: 14.8 ms
// compensating the chunks' sums only, 17.2 every term).
// Returns the ray sums in acc (alpha units).
// A x at 256^3 / 512^2 / 360 angles: 24.2 -> 12.9 ms, 24 -> 12.6 warp
// instructions per cell and 32 rays (two loads, one and a half packed FMA
// pairs and an add for the sums, two for t and the plane, the rest address and
// list), issue slots 67 % busy and L1 data wavefronts 54 %.
template <typename T, bool COMP, int R, bool OFF32, int DIR, bool CLAMP>
__device__ __forceinline__ void walk_cells(const DevGeom &g, const T *__restrict__ vol, CellList &cl, float amin,
                                           const RayZ (&z)[R], float4 *list, float (&acc)[R]) {
    constexpr int UNR = R == 2 ? 8 : 4;          // cells whose loads are in flight together
    float kb[R], kf[R], comp[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        float t = __fmaf_rn(amin, z[r].a, z[r].b);
        if (CLAMP) t = fminf(t, z[r].hi);
        kb[r] = __fadd_ru(t, z[r].m);
        kf[r] = kb[r] - z[r].m;
        comp[r] = 0.0f;
    }
    float ep = amin;
    bool last = false;
    const int maxchunks = (g.nx + g.ny) / CELL_CHUNK + 2;
    // voxel index k of the column: col - 1 + (bits(kb) - ZMAGIC_BITS) (up),
    // col - (bits(kb) - ZMAGIC_BITS) (down); the constant is added in the list
    constexpr unsigned UP = 0u - (unsigned)ZMAGIC_BITS - 1u, DOWN = (unsigned)ZMAGIC_BITS;
#pragma unroll 1
    for (int chunk = 0; chunk < maxchunks && !last; ++chunk) {
        const int n = cells_next(g, cl, DIR > 0 ? UP : DIR < 0 ? DOWN : 0u, (float2 *)list, &last);
        float s1[R], s2[R];                      // !COMP
#pragma unroll
        for (int r = 0; r < R; ++r) s1[r] = s2[r] = 0.0f;
#pragma unroll 1
        for (int c0 = 0; c0 < n; c0 += UNR) {
            float e[UNR];
            unsigned col[UNR];
#pragma unroll
            for (int p = 0; p < UNR / 2; ++p) {
                const float4 c2 = list[c0 / 2 + p];
                e[2 * p] = c2.x;
                col[2 * p] = __float_as_uint(c2.y);
                e[2 * p + 1] = c2.z;
                col[2 * p + 1] = __float_as_uint(c2.w);
            }
            float v[UNR][R], vn[UNR][R], w[UNR][R], len[UNR];
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                // DOWN + col stays below 2^32, so it is zero-extended; UP + col wraps to a negative index
                const T *base = DIR > 0 ? vol + (int64_t)(int)col[u] : vol + (int64_t)col[u];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int bits = __float_as_int(kb[r]);
                    const int step = DIR != 0 ? DIR : z[r].down ? -1 : 1;
                    const T *ptr;
                    if (OFF32) {
                        const unsigned c = DIR == 0 ? col[u] + (z[r].down ? DOWN : UP) : col[u];
                        ptr = (const T *)((const char *)vol + (size_t)((c + (unsigned)bits * (unsigned)step) * (unsigned)sizeof(T)));
                    } else {
                        ptr = base + (int64_t)bits * step;
                        if (DIR == 0) ptr += z[r].down ? (int64_t)ZMAGIC_BITS : -(int64_t)ZMAGIC_BITS - 1;
                    }
                    v[u][r] = Storage<T>::load(ptr);
                    vn[u][r] = Storage<T>::load(ptr + step);
                }
                len[u] = e[u] - ep;
                ep = e[u];
                const float2 e2 = make_float2(e[u], e[u]);
                if (R % 2 == 0) {
#pragma unroll
                    for (int r = 0; r + 1 < R; r += 2) {
                        float2 t = __ffma2_rn(e2, make_float2(z[r].a, z[r + 1].a), make_float2(z[r].b, z[r + 1].b));
                        if (CLAMP) t = make_float2(fminf(t.x, z[r].hi), fminf(t.y, z[r + 1].hi));
                        w[u][r] = __saturatef(t.x - kf[r]);
                        w[u][r + 1] = __saturatef(t.y - kf[r + 1]);
                        const float2 m2 = make_float2(z[r].m, z[r + 1].m);
                        const float2 k2 = __fadd2_ru(t, m2);
                        const float2 f2 = __ffma2_rn(m2, make_float2(-1.0f, -1.0f), k2);
                        kb[r] = k2.x;
                        kb[r + 1] = k2.y;
                        kf[r] = f2.x;
                        kf[r + 1] = f2.y;
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        float t = __fmaf_rn(e[u], z[r].a, z[r].b);
                        if (CLAMP) t = fminf(t, z[r].hi);
                        w[u][r] = __saturatef(t - kf[r]);
                        kb[r] = __fadd_ru(t, z[r].m);
                        kf[r] = kb[r] - z[r].m;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                if (R % 2 == 0) {
                    const float2 l2 = make_float2(len[u], len[u]), minus = make_float2(-1.0f, -1.0f);
#pragma unroll
                    for (int r = 0; r + 1 < R; r += 2) {
                        const float2 v2 = make_float2(v[u][r], v[u][r + 1]);
                        const float2 d2 = __ffma2_rn(v2, minus, make_float2(vn[u][r], vn[u][r + 1]));
                        if (COMP) {
                            const float2 wa = __fmul2_rn(make_float2(w[u][r], w[u][r + 1]), make_float2(z[r].inva, z[r + 1].inva));
                            const float2 a0 = make_float2(acc[r], acc[r + 1]);
                            const float2 y = __ffma2_rn(wa, d2, __ffma2_rn(l2, v2, make_float2(-comp[r], -comp[r + 1])));
                            const float2 t = __fadd2_rn(a0, y);
                            const float2 c2 = __ffma2_rn(y, minus, __ffma2_rn(a0, minus, t));
                            acc[r] = t.x;
                            acc[r + 1] = t.y;
                            comp[r] = c2.x;
                            comp[r + 1] = c2.y;
                            continue;
                        }
                        const float2 a1 = __ffma2_rn(l2, v2, make_float2(s1[r], s1[r + 1]));
                        const float2 a2 = __ffma2_rn(make_float2(w[u][r], w[u][r + 1]), d2, make_float2(s2[r], s2[r + 1]));
                        s1[r] = a1.x;
                        s1[r + 1] = a1.y;
                        s2[r] = a2.x;
                        s2[r + 1] = a2.y;
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float d = vn[u][r] - v[u][r];
                        if (COMP) {
                            const float y = __fmaf_rn(w[u][r] * z[r].inva, d, __fmaf_rn(len[u], v[u][r], -comp[r]));
                            const float t = acc[r] + y;
                            comp[r] = (t - acc[r]) - y;
                            acc[r] = t;
                            continue;
                        }
                        s1[r] = __fmaf_rn(len[u], v[u][r], s1[r]);
                        s2[r] = __fmaf_rn(w[u][r], d, s2[r]);
                    }
                }
            }
        }
        if (!COMP) {
#pragma unroll
            for (int r = 0; r < R; ++r)          // no ray parallel to the z planes has an s2
                acc[r] += z[r].a > 0.0f ? s1[r] + __fdividef(s2[r], z[r].a) : s1[r];
        }
    }
}

// Forward traversal of R rays of one detector column (DevGeom::zsingle):
// the walk for the warp's directions and z range.  list: 2 * CELL_CHUNK floats
// of shared memory of this warp.
template <typename T, bool COMP, int R, bool OFF32>
__device__ __forceinline__ void trace_rays_zsingle(const DevGeom &g, const T *__restrict__ vol, const RayAxis &rx,
                                                   const RayAxis &ry, const RayAxis (&rzax)[R], float4 *list,
                                                   float (&acc)[R]) {
    CellList cl;
    float amin;
    if (!cells_begin(g, rx, ry, cl, &amin)) return;
    bool up = false, down = false;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        up = up || rzax[r].I > 0.0f;
        down = down || rzax[r].I < 0.0f;
    }
    up = __any_sync(0xffffffffu, up);
    down = __any_sync(0xffffffffu, down);
    RayZ z[R];
    bool inside = true;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        z[r] = make_rayz(rzax[r], g.dz, g.nz, down && !up);
        inside = inside && __fmaf_rn(cl.amax, z[r].a, z[r].b) <= z[r].hi - ZPAST;
    }
    inside = __all_sync(0xffffffffu, inside);
    if (up && down)
        walk_cells<T, COMP, R, OFF32, 0, true>(g, vol, cl, amin, z, list, acc);
    else if (!down)
        inside ? walk_cells<T, COMP, R, OFF32, 1, false>(g, vol, cl, amin, z, list, acc)
               : walk_cells<T, COMP, R, OFF32, 1, true>(g, vol, cl, amin, z, list, acc);
    else
        inside ? walk_cells<T, COMP, R, OFF32, -1, false>(g, vol, cl, amin, z, list, acc)
               : walk_cells<T, COMP, R, OFF32, -1, true>(g, vol, cl, amin, z, list, acc);
}

// ------------------------------------------------------------- forward A x
//
// One tile = 8 warps = 8 adjacent detector columns (iu) x 32 R detector rows
// (iv) of one angle.  The volume is read in the padded z-fastest layout.
// Epilogue: proj = a * (A vol) + b * old (either projection layout), and one
// FP64 sums of squares of the stored values, one per warp, into
// partial_at()[warp] (when it returns non-null).  partial_at is called only in
// the epilogue, so that the address it computes is not held in a register
// through the traversal, and the sums need no block barrier (measured 6 %
// of the transpose's time with one).
// CELLS: the cell walk is compiled in (taken where DevGeom::zsingle).

// lists: FWD_COLS * FWD_LIST float4 of shared memory (the warps' cell lists).

constexpr int FWD_COLS = 8, FWD_THREADS = 32 * FWD_COLS;
constexpr int FWD_LIST = CELL_CHUNK / 2;         // float4 of one warp's cell list

template <typename T, bool COMP, int R, bool VFAST, bool OFF32, bool CELLS, typename PartialAt>
__device__ __forceinline__ void forward_tile(const DevGeom &g, const T *__restrict__ vol, T *__restrict__ proj,
                                             const Epilogue &epi, int tx, int ty, int a, PartialAt &&partial_at,
                                             float4 *lists) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int iu = tx * FWD_COLS + warp;
    const int iv0 = ty * 32 * R;
    const bool col_ok = iu < g.nu;            // uniform across the warp
    float acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0.0f;
    if (col_ok) {
        RayAxis rx, ry, rz[R];
        load_rays<R>(g, a, iu, iv0, g.nv, rx, ry, rz);
        if (CELLS && g.zsingle) {
            trace_rays_zsingle<T, COMP, R, OFF32>(g, vol, rx, ry, rz, lists + warp * FWD_LIST, acc);
        } else {
            // several z crossings per xy cell are possible: the exact
            // crossing-by-crossing traversal
            float comp[R];
#pragma unroll
            for (int r = 0; r < R; ++r) comp[r] = 0.0f;
            auto fetch = [&](int idx) { return Storage<T>::load(vol + idx); };
            auto seg = [&](int r, float len, float value) {
                const float term = len * value;
                if (COMP) {          // Kahan-compensated running sum
                    const float yk = term - comp[r];
                    const float t = acc[r] + yk;
                    comp[r] = (t - acc[r]) - yk;
                    acc[r] = t;
                } else {
                    acc[r] += term;
                }
            };
            trace_columns<R>(g, rx, ry, rz, 0, g.nx, 0, g.ny, 0, g.nz, (int)zf_col(g, 0, 0), g.nz + 2,
                             g.nx * (g.nz + 2), fetch, seg);
        }
    }
    double sq = 0.0;
    const double acoef = epi_a(epi), bcoef = epi_b(epi);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int iv = iv0 + r * 32 + lane;
        if (col_ok && iv < g.nv) {
            // output y[a][iu][iv] (v fastest: one warp writes consecutive rows) or y[a][iv][iu]
            const size_t ray = VFAST ? ((size_t)a * g.nu + iu) * g.nv + iv : ((size_t)a * g.nv + iv) * g.nu + iu;
            const float len = g.ray_len[(size_t)iu * g.nv + iv];
            double out = acoef * (double)(acc[r] * len);
            if (bcoef != 0.0) {
                const T *oldp = epi.old ? (const T *)epi.old : (const T *)proj;
                out += bcoef * (double)Storage<T>::ld_plain(oldp + ray);
            }
            const float stored = Storage<T>::round((float)out);
            Storage<T>::store(proj + ray, stored);
            if (VFAST && epi.weighted) epi.weighted[ray] = len * stored;
            sq += (double)stored * (double)stored;
        }
    }
    double *partial = partial_at();
    if (partial) warp_partial(sq, partial);
}

// ---------------------------------------------------------- transpose A^T y
//
// The tile for geometries that patch_tile.cuh does not take (steep cones, very
// coarse voxels) and for the shapes that have no patch form.  Gather form:
// each lane owns voxels (i, j, k) of one voxel column and sums len * w over
// every ray that meets them, in registers, angle by angle; the volume is
// written once (fused epilogue), so there are no atomics and the result does
// not depend on scheduling.  A warp owns one column (i, j) and 32 K consecutive
// k (k = k0 + kk * 32 + lane); a tile is 8 warps on a
// CX x (8 / CX) patch of columns.  For every angle the warp projects the
// cell's four corners to find the detector columns whose xy projection
// crosses cell (i, j), and each lane the detector rows that can meet its
// voxel's z slab (v = z dsd / depth over the corners' depths).  For each such
// column the warp takes the alpha interval [ain, aout] of the crossing (x and
// y plane crossings, warp-uniform), and a lane takes for each of its rows
// the segment
//     [max(ain, z entry), min(aout, z exit)].
// The z entry/exit of a row's ray in slab k does not depend on the angle
// (circular orbit), so it is read from the table DevGeom::zbox, which
// plane_alpha filled at geometry creation.
// Projections are read v-fastest and pre-weighted by the ray length:
// w[a][iu][iv] = |d'| * y.

constexpr int BWD_THREADS = 256;

// Calls body(iu, ain, aout) for every detector column iu in [iu0, iu1], in
// increasing order, whose ray column crosses voxel column (i, j) of angle a:
// [ain, aout] is the alpha interval of the x/y cell (warp-uniform), from the
// same plane_alpha values either way.  LANES: the lanes clip up to 32 columns
// at once (lane l: column c0 + l), then the warp walks them, taking each
// column's interval from its lane; otherwise the warp clips column by column
// (fewer registers).  All lanes must call it.
template <bool LANES, int UNROLL, typename Body>
__device__ __forceinline__ void for_crossing_columns(const DevGeom &g, int a, int i, int j, int iu0, int iu1,
                                                     int lane, Body &&body) {
    auto clip = [&](int iu, float &ain, float &aout) {
        const float4 xy = __ldg(&g.ray_xy[(size_t)a * g.nu + iu]);
        const float2 q = __ldg(&g.ray_xyq[(size_t)a * g.nu + iu]);
        ain = -FLT_MAX;
        aout = FLT_MAX;
        bool miss = false;
        clip_slab(RayAxis{xy.x, xy.y, q.x}, g.dx, i, i + 1, ain, aout, miss);
        clip_slab(RayAxis{xy.z, xy.w, q.y}, g.dy, j, j + 1, ain, aout, miss);
        if (miss) {
            ain = FLT_MAX;                             // empty: no crossing
            aout = -FLT_MAX;
        }
    };
    if (LANES) {
        for (int c0 = iu0; c0 <= iu1; c0 += 32) {
            const int cn = min(32, iu1 - c0 + 1);
            float cin = FLT_MAX, cout = -FLT_MAX;
            if (lane < cn) clip(c0 + lane, cin, cout);
#pragma unroll UNROLL
            for (int c = 0; c < cn; ++c) {
                const float ain = __shfl_sync(0xffffffffu, cin, c), aout = __shfl_sync(0xffffffffu, cout, c);
                if (ain < aout) body(c0 + c, ain, aout);
            }
        }
    } else {
#pragma unroll UNROLL
        for (int iu = iu0; iu <= iu1; ++iu) {
            float ain, aout;
            clip(iu, ain, aout);
            if (ain < aout) body(iu, ain, aout);
        }
    }
}

// Angles [a_begin, a_end) are summed in one call.  A scan whose projections
// do not fit in L2 is summed in passes over blocks of angles (launch_backward):
// `acc_in` (if not null) holds the FP32 sums of the earlier passes and
// `acc_out` (if not null) receives the running sums instead of the volume, so
// only the last pass applies the epilogue (with the FP64 sums of squares of
// the stored values into partial_at()[warp], when non-null, as in the
// forward tile).  Both are indexed
// ((j * nx + i) * nz + k) (unpadded); they may be the same buffer (each lane
// reads and writes only its own voxels).  ZFAST output goes to the padded
// z-fastest layout, else to the ABI layout x[k][j][i].
template <typename T, bool ZFAST, int CX, int K, int IU_UNROLL = 0, typename PartialAt>
__device__ __forceinline__ void backward_tile(const DevGeom &g, const float *__restrict__ wproj, T *__restrict__ vol,
                                              const Epilogue &epi, int tx, int ty, int tz, int a_begin, int a_end,
                                              const float *acc_in, float *acc_out, PartialAt &&partial_at) {
    constexpr int CY = 8 / CX;
    // detector columns clipped by the lanes at once (tiles of up to 2 voxels
    // per lane; the 4-voxel tiles keep the per-column clip, which needs fewer
    // registers) and columns per unrolled step of the column loops
    constexpr bool BWD_LANE_CLIP = K <= 2;
    constexpr int BWD_IU_UNROLL = IU_UNROLL > 0 ? IU_UNROLL : K == 2 ? 1 : 2;
    // The slab intervals of the candidate rows are loaded once per angle and
    // kept in registers (2 or 3 rows x 2 floats per voxel of the lane).
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = tx * CX + (warp % CX), j = ty * CY + (warp / CX);
    const int k0 = tz * 32 * K;
    const bool col_ok = i < g.nx && j < g.ny;          // uniform across the warp
    float acc[K];
#pragma unroll
    for (int kk = 0; kk < K; ++kk) {
        const int k = k0 + kk * 32 + lane;
        acc[kk] = acc_in && col_ok && k < g.nz ? acc_in[((size_t)j * g.nx + i) * g.nz + k] : 0.0f;
    }
    if (col_ok) {
        // The three candidate rows of each voxel start at its window's first
        // row moved down to fit the detector, and their slab intervals are
        // loaded once per angle (a row outside the window meets the voxel
        // nowhere and adds an exact zero).  The detector windows only select
        // candidates (every length is then computed exactly from the crossing
        // tables), so they use fast approximate divisions: their relative
        // error (~1e-6) stays far below the 0.05-pixel margins.
        const float inv_dv = 1.0f / g.dv, inv_du = 1.0f / g.du;
        const float cu = 0.5f * (g.nu - 1), cv = 0.5f * (g.nv - 1);
        float zlo[K], zhi[K];
        int zboff[K];
#pragma unroll
        for (int kk = 0; kk < K; ++kk) {
            const int k = k0 + kk * 32 + lane;
            zlo[kk] = (g.bz0 + k * g.dz) * inv_dv;
            zhi[kk] = (g.bz0 + (k + 1) * g.dz) * inv_dv;
            zboff[kk] = min(k, g.nz - 1) * g.nv;
        }
        const float x0 = g.bx0 + i * g.dx, x1 = x0 + g.dx;
        const float y0 = g.by0 + j * g.dy, y1 = y0 + g.dy;
        const size_t nuv = (size_t)g.nu * g.nv;
        for (int a = a_begin; a < a_end; ++a) {
            const float2 cs = __ldg(&g.trig[a]);
            float umin = FLT_MAX, umax = -FLT_MAX, magmin = FLT_MAX, magmax = 0.0f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float px = (c & 1) ? x1 : x0, py = (c & 2) ? y1 : y0;
                const float along = g.dso - (px * cs.x + py * cs.y);   // > 0: source outside
                const float mag = __fdividef(g.dsd, along);
                const float u = (-px * cs.y + py * cs.x) * mag;
                umin = fminf(umin, u);
                umax = fmaxf(umax, u);
                magmin = fminf(magmin, mag);
                magmax = fmaxf(magmax, mag);
            }
            const int iu0 = max(0, (int)ceilf(__fmaf_rn(umin, inv_du, cu - 0.05f)));
            const int iu1 = min(g.nu - 1, (int)floorf(__fmaf_rn(umax, inv_du, cu + 0.05f)));
            // rows 2 / 3: every lane's window has at most 2 / 3 rows
            int wlo[K];
            bool rows2 = true, rows3 = true;
#pragma unroll
            for (int kk = 0; kk < K; ++kk) {
                const int k = k0 + kk * 32 + lane;
                const float vmin = fminf(zlo[kk] * magmin, zlo[kk] * magmax);
                const float vmax = fmaxf(zhi[kk] * magmin, zhi[kk] * magmax);
                const int lo = max(0, (int)ceilf(vmin + (cv - 0.05f)));
                const int hi = k < g.nz ? min(g.nv - 1, (int)floorf(vmax + (cv + 0.05f))) : -1;
                rows2 = rows2 && hi - lo < 2;
                rows3 = rows3 && hi - lo < 3;
                wlo[kk] = lo;
            }
            rows2 = __all_sync(0xffffffffu, rows2) && g.nv >= 2;
            rows3 = __all_sync(0xffffffffu, rows3) && g.nv >= 3;
            const float *pa = wproj + (size_t)a * nuv;
            // A fixed sequence of ROWS rows per voxel, starting at the window's
            // first row moved down to fit the detector; their slab intervals
            // are loaded once per angle.
            auto short_pass = [&](auto rows_c) {
                constexpr int ROWS = decltype(rows_c)::value;
                int r0[K];
                float2 zb[K][ROWS];
#pragma unroll
                for (int kk = 0; kk < K; ++kk) {
                    r0[kk] = min(wlo[kk], g.nv - ROWS);
#pragma unroll
                    for (int t = 0; t < ROWS; ++t) zb[kk][t] = __ldg(&g.zbox[zboff[kk] + r0[kk] + t]);
                }
                // the column walk is unrolled by BWD_IU_UNROLL, so that the
                // next columns' loads are issued before this column's sums
                // (the per-column clip measured 7 % faster that way than the
                // compiler's choice, which kept the loop rolled; the lane
                // clip runs best rolled, at 3 CTAs per SM)
                for_crossing_columns<BWD_LANE_CLIP, BWD_IU_UNROLL>(g, a, i, j, iu0, iu1, lane, [&](int iu, float ain, float aout) {
                    const float *wcol = pa + (size_t)iu * g.nv;
#pragma unroll
                    for (int kk = 0; kk < K; ++kk) {
                        const float *wr = wcol + r0[kk];
#pragma unroll
                        for (int t = 0; t < ROWS; ++t) {
                            const float2 e = zb[kk][t];
                            const float lo = fmaxf(ain, e.x), hi = fminf(aout, e.y);
                            acc[kk] = __fmaf_rn(fmaxf(hi - lo, 0.0f), __ldg(wr + t), acc[kk]);
                        }
                    }
                });
            };
            if (rows2) {
                short_pass(std::integral_constant<int, 2>());
            } else if (rows3) {
                short_pass(std::integral_constant<int, 3>());
            } else {
                int rlo[K], rhi[K];
#pragma unroll
                for (int kk = 0; kk < K; ++kk) {
                    const int k = k0 + kk * 32 + lane;
                    const float vmin = fminf(zlo[kk] * magmin, zlo[kk] * magmax);
                    const float vmax = fmaxf(zhi[kk] * magmin, zhi[kk] * magmax);
                    rlo[kk] = max(0, (int)ceilf(vmin + (cv - 0.05f)));
                    rhi[kk] = k < g.nz ? min(g.nv - 1, (int)floorf(vmax + (cv + 0.05f))) : -1;
                }
                for_crossing_columns<BWD_LANE_CLIP, 1>(g, a, i, j, iu0, iu1, lane, [&](int iu, float ain, float aout) {
                    const float *wcol = pa + (size_t)iu * g.nv;
#pragma unroll
                    for (int kk = 0; kk < K; ++kk) {
                        for (int iv = rlo[kk]; iv <= rhi[kk]; ++iv) {
                            const float2 e = __ldg(&g.zbox[zboff[kk] + iv]);
                            const float lo = fmaxf(ain, e.x), hi = fminf(aout, e.y);
                            acc[kk] = __fmaf_rn(fmaxf(hi - lo, 0.0f), __ldg(wcol + iv), acc[kk]);
                        }
                    }
                });
            }
        }
    }
    if (acc_out) {                      // an earlier pass: keep the running sums
#pragma unroll
        for (int kk = 0; kk < K; ++kk) {
            const int k = k0 + kk * 32 + lane;
            if (col_ok && k < g.nz) acc_out[((size_t)j * g.nx + i) * g.nz + k] = acc[kk];
        }
        return;
    }
    const double acoef = epi_a(epi), bcoef = epi_b(epi);
    double sq = 0.0;
#pragma unroll
    for (int kk = 0; kk < K; ++kk) {
        const int k = k0 + kk * 32 + lane;
        if (!col_ok || k >= g.nz) continue;
        const size_t v = ZFAST ? (size_t)(zf_col(g, i, j) + k) : ((size_t)k * g.ny + j) * g.nx + i;
        double out = acoef * (double)acc[kk];
        if (bcoef != 0.0) {
            const T *oldp = epi.old ? (const T *)epi.old : (const T *)vol;
            out += bcoef * (double)Storage<T>::ld_plain(oldp + v);
        }
        const float stored = Storage<T>::round((float)out);
        Storage<T>::store(vol + v, stored);
        sq += (double)stored * (double)stored;
    }
    double *partial = partial_at();
    if (partial) warp_partial(sq, partial);
}

}  // namespace cbct
