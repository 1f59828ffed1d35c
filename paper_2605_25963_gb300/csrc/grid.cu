// grid.cu -- builds the uniform grids of grid.cuh on the device, once per mesh.
//
// A warp walks the cells of a triangle's box in a grid and keeps those that the triangle
// meets (separating axes, cells grown by kGridPad): a first pass counts, a prefix sum over
// the cells places the lists, a second pass fills them, and each list is put in the order
// of the triangle ids.  The distances to the nearest occupied cell follow axis by axis (the
// Chebyshev distance is separable).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <cstdlib>
#include <vector>

#include <cuda_runtime.h>

#include "gadep_internal.h"
#include "grid.cuh"

namespace gadep {

namespace {

constexpr double kGridPad = 0.02;           // of a cell, on every side
constexpr double kCellsPerTri = 160.0;
constexpr double kMinCells = 131072.0, kMaxCells = 4194304.0;  // per grid; indices stay below 2^23
// The fewest cells of all grids together, where there are more than 32: 200 small solids had
// 33e6 cells, which missed the caches (tracks on 200 boxes, 2e6 histories: trees 4.1 ms, 4.3
// with 2^17 cells to a solid, 3.3 now; building 11.5 -> 8.9 ms).
constexpr double kMinTotal = 4194304.0;
constexpr unsigned long long kMaxTotal = 1ull << 27;           // cells of all grids (2.4 GB while they are built)
constexpr int kMinTris = 2048, kMaxTris = 5 << 14;      // no run walks the grids of other meshes
constexpr int kMaxSkip = 64;
// The boxes of triangles in planes along the axes are flat, and a tree of such boxes finds a
// surface in few nodes: meshes with this share of them are left to the trees.  Trees / grids,
// megakernel, 3e5 histories at 122 keV: one box of 8,748 triangles 0.91, of 76,800 0.57, 8 boxes
// 0.87, 60 boxes 0.87, 6 nested boxes 1.06; cylinders 1.14 to 2.1.  (Coaxes have 0.1 to 0.6.)
constexpr double kMaxFlat = 0.8;
constexpr int kWarpCells = 4096;            // of a triangle's box, by one warp; larger boxes take more warps
// Cells of the triangles' boxes, on average over the triangles of all grids, at most.  Detectors
// have 200 to 600, lying obliquely 1,400; a tilted cylinder of 600 long triangles a side has
// 20,000 (2 x 0.6 ms, its trees 11).  Large triangles that lie obliquely have up to the 4e6 of
// a grid: 80,000 of them would take 4 s a pass (the trees 0.35), at this limit 60 ms.
constexpr double kMaxBox = 65536.0;

struct GridDesc {                           // host and build kernels
    double lo[3], s[3], inv[3];             // inv: 1 / s
    int n[3];
    uint32_t off;                           // first cell
};

// A triangle in a grid; the part of its box that a warp walks.
struct Pair { int32_t tri; uint16_t grid, part; };

// Whether the projections of triangle v on the axis (x, y) miss those of the box of half
// extent h round the origin.
__device__ __forceinline__ bool separated(const float v[3][3], int a, int b, float x, float y, float h)
{
    const float p0 = fmaf(v[0][a], x, v[0][b] * y), p1 = fmaf(v[1][a], x, v[1][b] * y), p2 = fmaf(v[2][a], x, v[2][b] * y);
    const float r = h * (fabsf(x) + fabsf(y));
    return fminf(p0, fminf(p1, p2)) > r || fmaxf(p0, fmaxf(p1, p2)) < -r;
}

// Entries of a list of c ids: rounded up to fours, one more for the length of a long one.
constexpr uint32_t kLong = 127;
__host__ __device__ inline uint32_t padded(uint32_t c) { return (c + (c >= kLong ? 4u : 3u)) & ~3u; }

// list null: counts[cell] += 1 per triangle that meets it; otherwise the ids go to
// list[start[cell] + counts[cell]++] (behind the length where the cell has kLong or more).
// One kernel for both, so that both find the same cells to the last bit.
// In FP32 and cells, with the triangle's lowest cell as the origin: coordinates of 160 are then
// good to 1e-5 of a cell, of 16,000 (the longest a thin region can be) to 1e-3, and kSlack and
// kGridPad cover that and the tests' rounding (the normal's, which a sliver's cancels, is added
// by itself): 0.2 % more cells than in FP64, none fewer.  Bound by issue, 2.5e11 cells of boxes a second.  FP64 throughout, a triangle to a
// warp, took 2.8 ms a pass on 3,456 triangles, most of it one warp with the largest box, and
// 3.1 on 20,088: now 0.14 and 0.29 (counting), 0.22 and 0.36 (lists).
constexpr float kSlack = 1e-3f;
__global__ void __launch_bounds__(256) raster_kernel(const Pair *pairs, long long n_pairs, const GridDesc *grids,
                                                     const float4 *tris, uint32_t *counts, const uint32_t *totals,
                                                     const uint32_t *start, uint32_t *list)
{
    const int lane = threadIdx.x & 31;
    const long long n_warps = (long long)gridDim.x * (blockDim.x >> 5);
    constexpr float h = 0.5f + (float)kGridPad + kSlack;
    for (long long p = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); p < n_pairs; p += n_warps) {
        const Pair pair = pairs[p];
        const GridDesc &g = grids[pair.grid];
        float v[3][3], far = 0.0f;
        int a0[3], na[3];
        const float4 q0 = tris[3 * (size_t)pair.tri], q1 = tris[3 * (size_t)pair.tri + 1], q2 = tris[3 * (size_t)pair.tri + 2];
        for (int a = 0; a < 3; ++a) {
            const double inv = g.inv[a];
            const double x0 = ((double)(a == 0 ? q0.x : (a == 1 ? q0.y : q0.z)) - g.lo[a]) * inv,
                         x1 = ((double)(a == 0 ? q1.x : (a == 1 ? q1.y : q1.z)) - g.lo[a]) * inv,
                         x2 = ((double)(a == 0 ? q2.x : (a == 1 ? q2.y : q2.z)) - g.lo[a]) * inv;
            a0[a] = max(1, (int)floor(fmin(x0, fmin(x1, x2)) - kGridPad));
            na[a] = min(g.n[a] - 2, (int)floor(fmax(x0, fmax(x1, x2)) + kGridPad)) - a0[a] + 1;
            v[0][a] = (float)(x0 - a0[a]);
            v[1][a] = (float)(x1 - a0[a]);
            v[2][a] = (float)(x2 - a0[a]);
            far = fmaxf(far, (float)na[a] + 1.0f);
        }
        float e[3][3], n[3], e2[2] = { 0.0f, 0.0f }, rn = 0.0f;
        for (int a = 0; a < 3; ++a) {
            e[0][a] = v[1][a] - v[0][a];
            e[1][a] = v[2][a] - v[1][a];
            e[2][a] = v[0][a] - v[2][a];
            e2[0] = fmaf(e[0][a], e[0][a], e2[0]);
            e2[1] = fmaf(e[1][a], e[1][a], e2[1]);
        }
        for (int a = 0; a < 3; ++a) {
            n[a] = e[0][(a + 1) % 3] * e[1][(a + 2) % 3] - e[0][(a + 2) % 3] * e[1][(a + 1) % 3];
            rn = fmaf(h, fabsf(n[a]), rn);
        }
        rn = fmaf(1e-6f * far, sqrtf(e2[0] * e2[1]), rn);
        const long long cells = (long long)na[0] * na[1] * na[2], first = (long long)pair.part * kWarpCells,
                        end = min(cells, first + kWarpCells);
        for (int i = (int)first + lane; i < (int)end; i += 32) {
            const int x = i % na[0], y = i / na[0] % na[1], z = i / (na[0] * na[1]);
            const float c[3] = { (float)x + 0.5f, (float)y + 0.5f, (float)z + 0.5f };
            float w[3][3];
            for (int k = 0; k < 3; ++k)
                for (int a = 0; a < 3; ++a) w[k][a] = v[k][a] - c[a];
            if (fabsf(fmaf(n[0], w[0][0], fmaf(n[1], w[0][1], n[2] * w[0][2]))) > rn) continue;
            bool apart = false;
            for (int k = 0; k < 3; ++k)
                apart = apart || separated(w, 1, 2, -e[k][2], e[k][1], h) || separated(w, 0, 2, e[k][2], -e[k][0], h) ||
                        separated(w, 0, 1, -e[k][1], e[k][0], h);
            if (apart) continue;
            const size_t cell = (size_t)g.off + ((size_t)(a0[2] + z) * g.n[1] + (a0[1] + y)) * g.n[0] + (a0[0] + x);
            const uint32_t at = atomicAdd(&counts[cell], 1u);
            if (list) list[start[cell] + (totals[cell] >= kLong ? 1u : 0u) + at] = (uint32_t)pair.tri;
        }
    }
}

constexpr int kScanBlock = 1024, kScanPer = 8, kScanTile = kScanBlock * kScanPer;

// Exclusive prefix sums of the padded list sizes within tiles of kScanTile cells; sums[tile] = tile total.
__global__ void __launch_bounds__(kScanBlock) scan_kernel(const uint32_t *in, uint32_t *out, unsigned long long n,
                                                          uint32_t *sums)
{
    __shared__ uint32_t s_warp[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long at = (unsigned long long)blockIdx.x * kScanTile + (unsigned long long)threadIdx.x * kScanPer;
    uint32_t v[kScanPer], sum = 0;
    for (int k = 0; k < kScanPer; ++k) { v[k] = at + k < n ? padded(in[at + k]) : 0u; sum += v[k]; }
    uint32_t inc = sum;
    for (int o = 1; o < 32; o <<= 1) { const uint32_t x = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += x; }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const uint32_t t = s_warp[lane];
        uint32_t x = t;
        for (int o = 1; o < 32; o <<= 1) { const uint32_t y = __shfl_up_sync(0xffffffffu, x, o); if (lane >= o) x += y; }
        s_warp[lane] = x - t;
        if (lane == 31) sums[blockIdx.x] = x;
    }
    __syncthreads();
    uint32_t pre = s_warp[warp] + inc - sum;
    for (int k = 0; k < kScanPer; ++k) { if (at + k < n) out[at + k] = pre; pre += v[k]; }
}

// Puts each list in the order of the ids (heap sort: a fan's centre may hold thousands)
// and writes the words of the occupied cells (one grid per blockIdx.y).  sums: of the lists'
// lengths and of their squares, per grid.
__global__ void __launch_bounds__(256) lists_kernel(const GridDesc *grids, const uint32_t *counts, const uint32_t *start,
                                                    uint32_t *list, int *cells, unsigned long long *sums)
{
    unsigned long long length = 0, square = 0;
    const GridDesc &g = grids[blockIdx.y];
    const uint32_t n = (uint32_t)g.n[0] * g.n[1] * g.n[2], first = n ? start[g.off] : 0u;
    for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const size_t i = (size_t)g.off + k;
        const uint32_t c = counts[i];
        if (!c) continue;
        length += c;
        square += (unsigned long long)c * c;
        uint32_t *l = list + start[i];
        if (c >= kLong) *l++ = c;
        for (uint32_t end = c, root = c / 2; end > 1u;) {
            uint32_t x;
            if (root > 0u) {
                x = l[--root];
            } else {
                x = l[--end];
                l[end] = l[0];
            }
            uint32_t at = root;
            while (2u * at + 1u < end) {
                uint32_t ch = 2u * at + 1u;
                if (ch + 1u < end && l[ch + 1u] > l[ch]) ++ch;
                if (l[ch] <= x) break;
                l[at] = l[ch];
                at = ch;
            }
            l[at] = x;
        }
        cells[i] = (int)(0x80000000u | min(c, kLong) << 24 | (start[i] - first) / 4u);
    }
    for (int o = 16; o > 0; o >>= 1) {
        length += __shfl_xor_sync(0xffffffffu, length, o);
        square += __shfl_xor_sync(0xffffffffu, square, o);
    }
    if ((threadIdx.x & 31) == 0 && length) {
        atomicAdd(&sums[2 * blockIdx.y], length);
        atomicAdd(&sums[2 * blockIdx.y + 1], square);
    }
}

__global__ void __launch_bounds__(256) offset_kernel(uint32_t *start, unsigned long long n, const uint32_t *tile_base)
{
    const unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) start[i] += tile_base[i / kScanTile];
}

// One axis of the distance to the nearest cell that is occupied or in the border
// layer: AXIS 0 from the counts, 1 and 2 from the distances of the axis before.
template <int AXIS>
__global__ void __launch_bounds__(256) distance_kernel(const GridDesc *grids, const uint32_t *counts, const uint8_t *in,
                                                       uint8_t *out, int *cells)
{
    const GridDesc &g = grids[blockIdx.y];
    const uint32_t n = (uint32_t)g.n[0] * g.n[1] * g.n[2];
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int x = (int)(i % g.n[0]), y = (int)(i / g.n[0] % g.n[1]), z = (int)(i / ((uint32_t)g.n[0] * g.n[1]));
        const size_t at = (size_t)g.off + i;
        const int here = AXIS == 0 ? x : (AXIS == 1 ? y : z), len = g.n[AXIS];
        const size_t step = AXIS == 0 ? 1 : (AXIS == 1 ? (size_t)g.n[0] : (size_t)g.n[0] * g.n[1]);
        const bool border = x == 0 || y == 0 || z == 0 || x == g.n[0] - 1 || y == g.n[1] - 1 || z == g.n[2] - 1;
        int d = border || counts[at] ? 0 : kMaxSkip;
        for (int j = 0; j < d; ++j)
            for (int sgn = -1; sgn <= 1; sgn += 2) {
                const int q = here + sgn * j;
                if (q < 0 || q >= len) { d = min(d, j); continue; }
                const size_t other = at + step * (size_t)(q - here);
                int v;
                if (AXIS == 0) v = q == 0 || q == len - 1 || counts[other] ? 0 : kMaxSkip;
                else v = in[other];
                d = min(d, max(j, v));
            }
        if (AXIS < 2) out[at] = (uint8_t)d;
        else if (border) cells[at] = 0;
        else if (!counts[at]) cells[at] = __float_as_int((float)d);
    }
}

// Records by mesh triangle id with the coordinates in the order (kx, ky, kz).
__global__ void __launch_bounds__(256) permute_kernel(const float4 *tris, int n_tri, float4 *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 3 * n_tri) return;
    const float4 v = tris[i];
    out[i] = make_float4(v.y, v.z, v.x, v.w);                             // kz = x: (y, z, x)
    out[(size_t)3 * n_tri + i] = make_float4(v.z, v.x, v.y, v.w);         // kz = y: (z, x, y)
    out[(size_t)6 * n_tri + i] = v;                                       // kz = z: (x, y, z)
}

template <class T>
cudaError_t alloc(T **p, size_t n)
{
    return cudaMalloc((void **)p, std::max<size_t>(n, 1) * sizeof(T));
}

}  // namespace

void grid_free(gadep_bvh *b)
{
    cudaFree(b->d_grid);
    cudaFree(b->d_grid_list);
    b->d_grid = b->d_grid_list = nullptr;
    b->grid_bytes = 0;
    b->grid_safe = b->grid_crowd = 0.0f;
}

// Builds the grids of b (device current).  Where they do not suit the mesh (coordinates
// too coarse for the cells' margin, lists too long for the cell words, too few or too many
// triangles, mostly flat or as large as the grids) or leave no memory, the tree serves
// alone; b->d_grid stays null.
gadep_status grid_build(gadep_bvh *b)
{
    const MeshData &m = b->geo;
    const int nt = m.n_tri();
    if (nt < kMinTris || nt > kMaxTris) return GADEP_OK;
    auto sets = region_triangle_sets(m);
    std::vector<int32_t> all((size_t)nt);
    for (int t = 0; t < nt; ++t) all[(size_t)t] = t;
    sets.push_back(all);
    const size_t ng = sets.size();
    std::vector<float> rec(12 * (size_t)nt);
    std::vector<float> low(3 * (size_t)nt, INFINITY), high(3 * (size_t)nt, -INFINITY);   // the triangles' boxes
    double far = 0.0;
    for (int t = 0; t < nt; ++t)
        for (int k = 0; k < 3; ++k) {
            for (int a = 0; a < 3; ++a) {
                const float x = (float)m.xyz[3 * (size_t)m.tri[3 * (size_t)t + k] + a];
                rec[12 * (size_t)t + 4 * k + a] = x;
                far = std::max(far, (double)std::fabs(x));
                low[3 * (size_t)t + a] = std::min(low[3 * (size_t)t + a], x);
                high[3 * (size_t)t + a] = std::max(high[3 * (size_t)t + a], x);
            }
            const int32_t w = k == 0 ? m.tri_solid[(size_t)t] + 1 : 0;
            std::memcpy(&rec[12 * (size_t)t + 4 * k + 3], &w, 4);
        }
    int flat = 0;
    for (int t = 0; t < nt; ++t) {
        const float *l = &low[3 * (size_t)t], *h = &high[3 * (size_t)t];
        const float thin = std::min(h[0] - l[0], std::min(h[1] - l[1], h[2] - l[2])),
                    wide = std::max(h[0] - l[0], std::max(h[1] - l[1], h[2] - l[2]));
        flat += thin <= 1e-3f * wide;
    }
    if (flat > kMaxFlat * nt) return GADEP_OK;
    std::vector<GridDesc> desc(ng);
    std::vector<Pair> pairs;
    unsigned long long total = 0;
    double pad = INFINITY, left = 0.0;       // cells of boxes that may still come
    for (const auto &set : sets) left += kMaxBox * (double)set.size();
    for (size_t r = 0; r < ng; ++r) {
        GridDesc &g = desc[r];
        std::memset(&g, 0, sizeof(g));
        g.off = (uint32_t)total;
        if (sets[r].empty()) continue;
        double lo[3] = { INFINITY, INFINITY, INFINITY }, hi[3] = { -INFINITY, -INFINITY, -INFINITY };
        for (int32_t t : sets[r])
            for (int a = 0; a < 3; ++a) {
                lo[a] = std::min(lo[a], (double)low[3 * (size_t)t + a]);
                hi[a] = std::max(hi[a], (double)high[3 * (size_t)t + a]);
            }
        double vol = 1.0, longest = 0.0;
        for (int a = 0; a < 3; ++a) longest = std::max(longest, hi[a] - lo[a]);
        for (int a = 0; a < 3; ++a) vol *= std::max(hi[a] - lo[a], 1e-3 * longest);
        const double least = std::min(kMinCells, kMinTotal / (double)ng);
        const double want = std::min(std::max(kCellsPerTri * (double)sets[r].size(), least), kMaxCells);
        for (double s = std::cbrt(vol / want);; s *= 1.02) {
            double cells = 1.0;
            for (int a = 0; a < 3; ++a) {
                const double n = std::floor((hi[a] - lo[a]) / s + 0.1) + 3.0;   // a border cell on each side
                g.n[a] = (int)std::min(n, 1e6);
                g.s[a] = s;
                g.inv[a] = 1.0 / s;
                g.lo[a] = 0.5 * (lo[a] + hi[a]) - 0.5 * g.n[a] * s;
                cells *= n;
            }
            if (cells <= kMaxCells) break;
        }
        pad = std::min(pad, kGridPad * g.s[0]);
        // a box has at most two cells more along each axis than its length goes into whole ones
        for (int32_t t : sets[r]) {
            double box = 1.0;
            for (int a = 0; a < 3; ++a)
                box *= std::min((high[3 * (size_t)t + a] - low[3 * (size_t)t + a]) * g.inv[a] + 3.0, (double)g.n[a]);
            if ((left -= box) < 0.0) return GADEP_OK;
            for (int part = 0; part * (double)kWarpCells < box; ++part)
                pairs.push_back(Pair{ t, (uint16_t)r, (uint16_t)part });
        }
        total += (unsigned long long)g.n[0] * g.n[1] * g.n[2];
    }
    // the rounding of a position |x| away from the coordinate origin is a few units of
    // 2^-24 |x|: half the pad covers 16 of them up to this distance
    const double safe = 0.5 * pad * 16777216.0 / 16.0;
    if (!(far < 0.25 * safe) || total > kMaxTotal) return GADEP_OK;
    // device blocks: descriptors, cells and permuted triangles; the lists, whose size
    // the counting pass gives
    const size_t o_cells = (ng * 64 + 255) & ~(size_t)255;
    const size_t o_tris = o_cells + (((size_t)total * 4 + 255) & ~(size_t)255);
    char *base = nullptr;
    GridDesc *d_desc = nullptr;
    Pair *d_pairs = nullptr;
    uint32_t *counts = nullptr, *cursor = nullptr, *start = nullptr, *sums = nullptr, *list = nullptr;
    uint8_t *dist = nullptr;
    unsigned long long *lengths = nullptr;
    float4 *tris = nullptr;
    const uint32_t tiles = (uint32_t)((total + kScanTile - 1) / kScanTile);
    cudaError_t e = alloc(&base, o_tris + (size_t)nt * 9 * sizeof(float4));
    if (e == cudaSuccess) e = alloc(&d_desc, ng);
    if (e == cudaSuccess) e = alloc(&d_pairs, pairs.size());
    if (e == cudaSuccess) e = alloc(&counts, total);
    if (e == cudaSuccess) e = alloc(&cursor, total);
    if (e == cudaSuccess) e = alloc(&start, total);
    if (e == cudaSuccess) e = alloc(&sums, tiles);
    if (e == cudaSuccess) e = alloc(&dist, 2 * total);
    if (e == cudaSuccess) e = alloc(&tris, (size_t)nt * 3);
    if (e == cudaSuccess) e = alloc(&lengths, 2 * ng);
    if (e == cudaSuccess) e = cudaMemcpy(d_desc, desc.data(), ng * sizeof(GridDesc), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(d_pairs, pairs.data(), pairs.size() * sizeof(Pair), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(tris, rec.data(), rec.size() * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(counts, 0, total * 4);
    if (e == cudaSuccess) e = cudaMemset(cursor, 0, total * 4);
    if (e == cudaSuccess) e = cudaMemset(lengths, 0, 2 * ng * sizeof(*lengths));
    int *cells = (int *)(base + o_cells);
    const int blocks = (int)std::min<size_t>(65535, (pairs.size() + 7) / 8);
    const unsigned cell_blocks = (unsigned)((total + 255) / 256);
    std::vector<uint32_t> tile(tiles), first(ng + 1);
    std::vector<unsigned long long> sum(2 * ng, 0);
    unsigned long long entries = 0;
    bool fits = true;
    if (e == cudaSuccess) {
        raster_kernel<<<blocks, 256>>>(d_pairs, (long long)pairs.size(), d_desc, tris, counts, nullptr, nullptr, nullptr);
        scan_kernel<<<tiles, kScanBlock>>>(counts, start, total, sums);
        e = cudaMemcpy(tile.data(), sums, tiles * 4, cudaMemcpyDeviceToHost);
        for (uint32_t &t : tile) {
            const uint32_t n = t;
            t = (uint32_t)entries;
            entries += n;
        }
        fits = entries < (1ull << 31);
        first[ng] = (uint32_t)entries;
        if (e == cudaSuccess && fits) {
            e = cudaMemcpy(sums, tile.data(), tiles * 4, cudaMemcpyHostToDevice);
            offset_kernel<<<cell_blocks, 256>>>(start, total, sums);
            // the first list entry of every grid; a cell word counts fours from it in 24 bits
            for (size_t r = ng; r-- > 0 && e == cudaSuccess;) {
                first[r] = first[r + 1];
                if (desc[r].n[0]) e = cudaMemcpy(&first[r], start + desc[r].off, 4, cudaMemcpyDeviceToHost);
                fits = fits && first[r + 1] - first[r] < (1u << 26);
            }
        }
    }
    if (e == cudaSuccess && fits) {
        std::vector<float> gd(16 * ng, 0.0f);
        for (size_t r = 0; r < ng; ++r) {
            float *f = &gd[16 * r];
            for (int a = 0; a < 3; ++a) {
                f[a] = (float)desc[r].lo[a];
                f[4 + a] = (float)desc[r].s[a];
                f[8 + a] = desc[r].n[0] ? (float)(1.0 / desc[r].s[a]) : 0.0f;
                f[12 + a] = (float)desc[r].n[a];
            }
            std::memcpy(&f[3], &desc[r].off, 4);
            std::memcpy(&f[7], &first[r], 4);
        }
        e = cudaMemcpy(base, gd.data(), gd.size() * 4, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = alloc(&list, (size_t)entries);
        if (e == cudaSuccess) {
            const dim3 by_grid(512, (unsigned)ng);
            raster_kernel<<<blocks, 256>>>(d_pairs, (long long)pairs.size(), d_desc, tris, cursor, counts, start, list);
            lists_kernel<<<by_grid, 256>>>(d_desc, counts, start, list, cells, lengths);
            distance_kernel<0><<<by_grid, 256>>>(d_desc, counts, nullptr, dist, nullptr);
            distance_kernel<1><<<by_grid, 256>>>(d_desc, counts, dist, dist + total, nullptr);
            distance_kernel<2><<<by_grid, 256>>>(d_desc, counts, dist + total, nullptr, cells);
            permute_kernel<<<(3 * nt + 255) / 256, 256>>>(tris, nt, (float4 *)(base + o_tris));
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpy(sum.data(), lengths, sum.size() * sizeof(sum[0]), cudaMemcpyDeviceToHost);
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
    }
    cudaFree(d_desc);
    cudaFree(d_pairs);
    cudaFree(counts);
    cudaFree(cursor);
    cudaFree(start);
    cudaFree(sums);
    cudaFree(dist);
    cudaFree(tris);
    cudaFree(lengths);
    if (e != cudaSuccess || !list) {
        cudaFree(base);
        cudaFree(list);
        if (e != cudaSuccess && e != cudaErrorMemoryAllocation)
            return fail(GADEP_E_CUDA, "gadep_bvh_build: grids: %s", cudaGetErrorString(e));
        cudaGetLastError();
        return GADEP_OK;
    }
    b->d_grid = base;
    b->d_grid_list = list;
    b->grid_cells = o_cells;
    b->grid_tris = o_tris;
    b->grid_bytes = o_tris + (size_t)nt * 9 * sizeof(float4) + (size_t)entries * sizeof(uint32_t);
    b->grid_safe = (float)safe;
    b->grid_crowd = 0.0f;
    for (size_t r = 0; r + 1 < ng; ++r)             // the grid of every triangle serves few queries
        if (sum[2 * r]) b->grid_crowd = std::max(b->grid_crowd, (float)((double)sum[2 * r + 1] / (double)sum[2 * r]));
    return GADEP_OK;
}

// The grids as the kernels take them (desc null: none were built).
dev::GridSet grid_set(const gadep_bvh *b)
{
    dev::GridSet g{};
    if (!b->d_grid) return g;
    const char *base = (const char *)b->d_grid;
    g.desc = (const float4 *)base;
    g.cells = (const int *)(base + b->grid_cells);
    g.tris = (const float4 *)(base + b->grid_tris);
    g.list = (const uint32_t *)b->d_grid_list;
    g.n_tri = b->geo.n_tri();
    g.all = (int)(b->regions.size() / 4);
    return g;
}

}  // namespace gadep
