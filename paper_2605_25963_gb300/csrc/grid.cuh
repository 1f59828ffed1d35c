// grid.cuh -- uniform-grid walk of the segment queries (built by grid.cu).
//
// Every region's triangle set (its own solid's and its child solids' surfaces) and
// the set of every triangle has a uniform grid of its own.  A cell's word is
//   0            the border layer: the walk leaves the grid;
//   > 0          an empty cell, the bits of a float r: every cell nearer than r cells
//                (Chebyshev distance) is empty and inside the grid, so the walk may
//                leave the cube of those cells in one step;
//   < 0          the cell's list of mesh triangle ids: its length in bits 24..30 (127:
//                the length is the list's first entry), its start in bits 0..23, in
//                fours of entries from the grid's first list entry.
//
// Why a grid beside the tree of device_common.cuh: most queries of a photon are short
// hops between the thin nested shells of a detector.  A tree descends from its root to
// the leaf that the ray starts in whatever the length of the hop (coax: 8.6 wide nodes
// of ~130 instructions and 7.4 triangle tests per query); the grid starts in the cell of
// the ray's position and is done in a few cells of ~60 instructions.
//
// Robustness: a triangle is listed in every cell that it meets when the cell is grown
// by kGridPad of its size on all sides, which exceeds the rounding of the positions
// computed here for origins within gadep_bvh::grid_safe of the coordinate origin (callers
// use the tree beyond that).  The cell indices are carried as exact small floats and
// only ever move forward, by at least one cell per step, and no step passes the
// border layer, so a walk ends after at most nx + ny + nz steps.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "device_common.cuh"

namespace gadep {
namespace dev {

// Triangle records by mesh triangle id, once per dominant axis kz of the ray: three
// float4 (v0, region id), (v1, -), (v2, -) with the coordinates in the order
// (kx, ky, kz), so that one triangle test serves every axis without selects.
struct GridSet {
    const float4 *desc;       // four float4 per grid: (lo, first cell), (cell size, first list
                              // entry), (1 / cell size, -), (cells per axis, 0 = empty grid; -).
                              // Null: no grids
    const int *cells;
    const uint32_t *list;
    const float4 *tris;       // [3][n_tri][3]
    int n_tri;
    int all;                  // grid of every triangle
};

// One walk: per axis mirrored so that the ray moves towards larger cells.
struct Walk {
    float cx, cy, cz;         // cell
    float ox, oy, oz;         // origin in cells
    float dx, dy, dz;         // cells per mm
    float ix, iy, iz;         // mm per cell
    float sx, sy, sz, base;   // index of a cell = sx cx + sy cy + sz cz + base - 2^23
    uint32_t off;             // first cell of the grid - bits of 2^23
};

constexpr float kIndexBias = 8388608.0f;      // 2^23: the index in the low mantissa bits

__device__ __forceinline__ void walk_axis(float lo, float s, float inv, float n, float stride, float o, float d,
                                          float &om, float &dm, float &im, float &st, float &base, float &low,
                                          float &tin, float &tout)
{
    const bool neg = d < 0.0f;
    const float g = (o - lo) * inv;
    const float ad = fmaxf(fabsf(d), 1e-30f);
    om = neg ? -g : g;
    dm = ad * inv;
    im = __fdividef(s, ad);
    low = neg ? 1.0f - n : 1.0f;                       // the border layer is left out
    st = neg ? -stride : stride;
    base = neg ? base - stride : base;                 // mirrored cell c stands for -(c + 1)
    tin = fmaxf(tin, (low - om) * im);
    tout = fminf(tout, (low + (n - 2.0f) - om) * im);
}

__device__ __forceinline__ int walk_word(const Walk &w, const int *__restrict__ cells)
{
    const float f = fmaf(w.cx, w.sx, fmaf(w.cy, w.sy, fmaf(w.cz, w.sz, w.base)));
    return __ldg(cells + (w.off + __float_as_uint(f)));
}

__device__ __forceinline__ float floor_cell(float x)
{
    return __fadd_rd(x, 12582912.0f) - 12582912.0f;    // exact floor for |x| < 2^22
}

// Starts a walk of grid g at distance t0 along the ray; returns the first cell's word
// (0: the ray does not meet the grid beyond t0, or is not finite) and the grid's first
// list entry.
__device__ __forceinline__ int walk_begin(Walk &w, const GridSet &G, int g, float ox, float oy, float oz, float dx,
                                          float dy, float dz, float t0, uint32_t &lists)
{
    const float4 a = __ldg(G.desc + 4 * g), s = __ldg(G.desc + 4 * g + 1), v = __ldg(G.desc + 4 * g + 2),
                 n = __ldg(G.desc + 4 * g + 3);
    lists = __float_as_uint(s.w);
    if (n.x == 0.0f) return 0;
    w.off = __float_as_uint(a.w) - __float_as_uint(kIndexBias);
    w.base = kIndexBias;
    float tin = t0, tout = INFINITY, lx, ly, lz;
    walk_axis(a.x, s.x, v.x, n.x, 1.0f, ox, dx, w.ox, w.dx, w.ix, w.sx, w.base, lx, tin, tout);
    walk_axis(a.y, s.y, v.y, n.y, n.x, oy, dy, w.oy, w.dy, w.iy, w.sy, w.base, ly, tin, tout);
    walk_axis(a.z, s.z, v.z, n.z, n.x * n.y, oz, dz, w.oz, w.dz, w.iz, w.sz, w.base, lz, tin, tout);
    // min and max drop NaN operands; the sum keeps them
    const float sum = w.ox + w.oy + w.oz + w.dx + w.dy + w.dz + tin;
    if (!(tin <= tout && fabsf(sum) < INFINITY)) return 0;
    w.cx = fminf(fmaxf(floor_cell(fmaf(tin, w.dx, w.ox)), lx), lx + (n.x - 3.0f));
    w.cy = fminf(fmaxf(floor_cell(fmaf(tin, w.dy, w.oy)), ly), ly + (n.y - 3.0f));
    w.cz = fminf(fmaxf(floor_cell(fmaf(tin, w.dz, w.oz)), lz), lz + (n.z - 3.0f));
    return walk_word(w, G.cells);
}

// Leaves the cube of cells nearer than r (1: the cell itself).  Returns the distance at
// which the ray leaves it and moves the walk to the cell behind.
__device__ __forceinline__ float walk_step(Walk &w, float r)
{
    const float px = w.cx + r, py = w.cy + r, pz = w.cz + r;
    const float tx = (px - w.ox) * w.ix, ty = (py - w.oy) * w.iy, tz = (pz - w.oz) * w.iz;
    const float te = fminf(tx, fminf(ty, tz));
    // the axis that is left moves to its plane, the others to the ray's position
    w.cx = fmaxf(tx <= te ? px : w.cx, floor_cell(fmaf(te, w.dx, w.ox)));
    w.cy = fmaxf(ty <= te ? py : w.cy, floor_cell(fmaf(te, w.dy, w.oy)));
    w.cz = fmaxf(tz <= te ? pz : w.cz, floor_cell(fmaf(te, w.dz, w.oz)));
    return te;
}

// Shear of a ray for the triangle test on permuted records (see tri_test in
// device_common.cuh): the origin in the order (kx, ky, kz), never swapped; flip = d[kz] < 0.
struct GridRay {
    float ox, oy, oz;
    float sx, sy, sz;
    bool flip;
    const float4 *tris;
};

__device__ __forceinline__ int dominant_axis(float dx, float dy, float dz)
{
    const float ax = fabsf(dx), ay = fabsf(dy), az = fabsf(dz);
    return (ax > ay) ? ((ax > az) ? 0 : 2) : ((ay > az) ? 1 : 2);
}

__device__ __forceinline__ GridRay grid_ray(const GridSet &G, const ShearK &sh, float ox, float oy, float oz)
{
    GridRay r;
    r.ox = sh.kz == 2 ? ox : (sh.kz == 0 ? oy : oz);
    r.oy = sh.kz == 2 ? oy : (sh.kz == 0 ? oz : ox);
    r.oz = sh.kz == 2 ? oz : (sh.kz == 0 ? ox : oy);
    r.sx = sh.sx; r.sy = sh.sy; r.sz = sh.sz;
    r.flip = sh.flip;
    r.tris = G.tris + (size_t)(3 * sh.kz) * G.n_tri;
    return r;
}

// The list of a cell word: first entry and length.
__device__ __forceinline__ uint32_t cell_list(const uint32_t *__restrict__ list, uint32_t lists, int word, uint32_t &n)
{
    uint32_t at = lists + 4u * ((uint32_t)word & 0xffffffu);
    n = ((uint32_t)word >> 24) & 127u;
    if (n == 127u) n = __ldg(list + at++);
    return at;
}

// The nearest hit so far of a query.  Its distance is kept as the fraction of the
// edge-function test and, to about 2^-21, as a number: the division is carried out only
// where two distances are too close for the numbers to order them.
struct Nearest {
    float t, num, den;
    int best;                  // mesh triangle id << 1 | entering, -1 = none; kTied set when
                               // another triangle lies at exactly the same distance
};
constexpr int kTied = 1 << 30;

// The edge functions in FP64, whose products of binary32 values are exact.  Out of line:
// inlined, ptxas ran the FP64 instructions in every test under a predicate, and the FP64
// pipe, at 84 % of its rate, made the trace kernel four times slower.
static __device__ __noinline__ float3 exact_edges(float Ax, float Ay, float Bx, float By, float Cx, float Cy)
{
    return make_float3((float)__dsub_rn(__dmul_rn((double)Cx, (double)By), __dmul_rn((double)Cy, (double)Bx)),
                       (float)__dsub_rn(__dmul_rn((double)Ax, (double)Cy), __dmul_rn((double)Ay, (double)Cx)),
                       (float)__dsub_rn(__dmul_rn((double)Bx, (double)Ay), __dmul_rn((double)By, (double)Ax)));
}

// The watertight test of tri_test_k (device_common.cuh), operation for operation, on the
// permuted record of triangle id; o: origin (kx, ky, kz), t_min; s: shear, first record
// of the ray's axis | flip << 31.  A hit's distance is left as the fraction num / den.
__device__ __forceinline__ bool grid_tri_test(const GridSet &G, const float4 &o, const float4 &s, int id, float &num,
                                              float &den)
{
    const float4 *q = G.tris + ((__float_as_uint(s.w) & 0x7fffffffu) + 3u * (uint32_t)id);
    const float4 a = __ldg(q), b = __ldg(q + 1), c = __ldg(q + 2);
    const float Akz = a.z - o.z, Bkz = b.z - o.z, Ckz = c.z - o.z;
    const float Ax = fmaf(-s.x, Akz, a.x - o.x), Ay = fmaf(-s.y, Akz, a.y - o.y);
    const float Bx = fmaf(-s.x, Bkz, b.x - o.x), By = fmaf(-s.y, Bkz, b.y - o.y);
    const float Cx = fmaf(-s.x, Ckz, c.x - o.x), Cy = fmaf(-s.y, Ckz, c.y - o.y);
    float U = __fsub_rn(__fmul_rn(Cx, By), __fmul_rn(Cy, Bx));
    float V = __fsub_rn(__fmul_rn(Ax, Cy), __fmul_rn(Ay, Cx));
    float W = __fsub_rn(__fmul_rn(Bx, Ay), __fmul_rn(By, Ax));
    if (fminf(fabsf(U), fminf(fabsf(V), fabsf(W))) == 0.0f) {
        const float3 e = exact_edges(Ax, Ay, Bx, By, Cx, Cy);
        U = e.x; V = e.y; W = e.z;
    }
    den = U + V + W;
    if (den == 0.0f || (fminf(U, fminf(V, W)) < 0.0f && fmaxf(U, fmaxf(V, W)) > 0.0f)) return false;
    num = U * (s.z * Akz) + V * (s.z * Bkz) + W * (s.z * Ckz);
    return true;
}

// Takes the hit num / den on triangle id when it lies beyond t_min and before h: the
// hits taken are those that the rounded quotients would select.  Which of two triangles
// at the same quotient (a ray through their common edge) is taken depends on the order of
// the tests; the caller asks the tree then, whose order has always decided.
__device__ __forceinline__ void nearer(Nearest &h, float num, float den, int id, bool flip, float t_min)
{
    const float t = __fdividef(num, den);
    const float lo = t * (1.0f - 1e-6f), hi = t * (1.0f + 1e-6f);
    bool take = lo > t_min && hi < h.t;
    if (!take && !(hi <= t_min || lo >= h.t)) {
        const float x = num / den, y = h.num / h.den;
        take = x > t_min && x < y;
        if (x > t_min && x == y && h.best >= 0 && ((h.best & (kTied - 1)) >> 1) != id) h.best |= kTied;
    }
    if (take) {
        h.t = t;
        h.num = num;
        h.den = den;
        h.best = (id << 1) | ((den > 0.0f) != flip ? 1 : 0);
    }
}

// plane_t (device_common.cuh) of hit h, the quotient of its fraction taken only where the
// plane's distance cannot be.
__device__ __forceinline__ float nearest_t(const float4 *__restrict__ planes, const Nearest &h, float ox, float oy,
                                           float oz, float dx, float dy, float dz, float t_min)
{
    const float4 p = __ldg(planes + ((h.best & (kTied - 1)) >> 1));
    const float dn = fmaf(p.x, dx, fmaf(p.y, dy, p.z * dz));
    const float num = fmaf(-p.x, ox, fmaf(-p.y, oy, fmaf(-p.z, oz, p.w)));
    const float t = num / dn;
    return (isfinite(t) && t > t_min) ? t : h.num / h.den;
}

// A direction component back from its reciprocal, as the tree's queries take it for the
// plane distance: both forms then give the same bits.
__device__ __forceinline__ float back_from_reciprocal(float d)
{
    return __frcp_rn(1.0f / (fabsf(d) > 1e-30f ? d : copysignf(1e-30f, d)));
}

// Nearest triangle of grid g along o + t d with t_min < t < t_max (exclusive), skipping
// mesh triangle `exclude`: its mesh triangle id or -1; t_hit and entering set on a hit.
// The selection and the distance are those of traverse() in device_common.cuh, but where
// two triangles tie for the nearest hit, whose order of tests decides: such queries are
// left to the tree (`left` set, no hit).  t_min >= 0.
template <bool COUNT>
__device__ __forceinline__ int grid_query(const GridSet &G, const float4 *__restrict__ planes, int g, float ox, float oy,
                                          float oz, float dx, float dy, float dz, float t_min, int exclude,
                                          float &t_hit, bool &entering, bool &left, TravStats &st,
                                          float t_max = INFINITY)
{
    left = false;
    Walk w;
    uint32_t lists;
    int word = walk_begin(w, G, g, ox, oy, oz, dx, dy, dz, t_min, lists);
    if (word == 0) return -1;
    const GridRay r = grid_ray(G, make_shear_k(dx, dy, dz), ox, oy, oz);
    const float4 o = make_float4(r.ox, r.oy, r.oz, t_min);
    const float4 s = make_float4(r.sx, r.sy, r.sz, __uint_as_float((uint32_t)(r.tris - G.tris)));
    Nearest h{ t_max, t_max, 1.0f, -1 };
    uint32_t nn = 0, nt = 0;
    while (true) {
        float skip = __int_as_float(word);
        ++nn;
        if (word < 0) {
            uint32_t n;
            const uint32_t at = cell_list(G.list, lists, word, n);
            for (uint32_t k = 0; k < n; ++k) {
                const int id = (int)__ldg(G.list + at + k);
                if (id == exclude) continue;
                ++nt;
                float num, den;
                if (grid_tri_test(G, o, s, id, num, den)) nearer(h, num, den, id, r.flip, t_min);
            }
            skip = 1.0f;
        }
        if (walk_step(w, skip) >= h.t) break;
        word = walk_word(w, G.cells);
        if (word == 0) break;
    }
    if (COUNT) { st.nodes += nn; st.boxes += nn; st.tris += nt; }
    if (h.best < 0) return -1;
    if ((h.best & kTied) != 0) {
        left = true;
        return -1;
    }
    t_hit = nearest_t(planes, h, ox, oy, oz, back_from_reciprocal(dx), back_from_reciprocal(dy),
                      back_from_reciprocal(dz), t_min);
    entering = (h.best & 1) != 0;
    return h.best >> 1;
}

}  // namespace dev
}  // namespace gadep
