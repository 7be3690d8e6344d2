// Initial particles of a body (Sec. 3.2), on the device.
//
// Compiled with -fmad=false: the ray-parity arithmetic is evaluated exactly
// in the written order, so inside / outside is decided as by any other IEEE
// implementation of the same formulas.
// Cell sets are bitmaps of rows padded to whole words: bit x & 31 of word
// (x >> 5) + W (y + ny z), W = ceil(nx / 32), so that a word is 32 columns or
// 32 cells of a row, and words in order are cells in key order.  Work that
// belongs to the surface runs over the occupied cells only (C_compact).
//   k_crossings      +z rays of Fig. 6 from the cell centres of every column
//                    (displaced by (1.234567e-6, 2.345678e-6) dx in x, y so
//                    they meet no edge or vertex exactly) against the
//                    triangles of the occupied cells, each triangle once per
//                    column: a crossing toggles the cells below it, noted at
//                    the highest one
//   k_inside_words   the parity of the crossings above every cell, 32 columns
//                    at a time (exclusive or down the columns)
//   k_dilate_x/_yz   Chebyshev distance <= band to a cell with triangles, by
//                    three one-axis dilations
//   k_surface_cells  a cell with triangles maps its centre to the nearest
//                    triangle of the cell whose foot is inside (else it is
//                    discarded, Fig. 9b)
//   k_word_counts    surface cells and empty inside cells per word; their
//                    scan gives the particles' places in key order
//   k_emit_surface, k_emit_volume
// A body of C cells moves C / 8 bytes a pass instead of C to 4 C: the gear
// turned in space (1.7e8 cells, 2.9 M particles) 12.0 -> 0.5 ms of kernels, the
// largest k_crossings (0.13 ms).
#include <cfloat>
#include <cmath>

#include "body.h"

namespace fppg {
namespace {

constexpr uint32_t kColEntries = 256;   // crossed triangle entries a column may hold

__device__ inline bool bit_of(const uint32_t *m, uint64_t c) { return (m[c >> 5] >> (c & 31u)) & 1u; }

struct MapGrid {
    float o[3];
    int n[3];
    int W;                 // words of a row
    double dx;
    const float *mid[3];   // cell centres along each axis (k_centres)
    uint32_t hash_mask;
    float edge_tol;
};

// the cell centres along the axes, evaluated in FP64 once instead of by every
// cell (the FP64 units are far slower than the rest of this path)
__global__ void __launch_bounds__(256) k_centres(MapGrid g, float *__restrict__ out) {
    const int i = blockIdx.x * 256 + threadIdx.x;
    const int a = i < g.n[0] ? 0 : i < g.n[0] + g.n[1] ? 1 : 2;
    const int k = i - (a > 0 ? g.n[0] : 0) - (a > 1 ? g.n[1] : 0);
    if (k < g.n[a]) out[i] = (float)((double)g.o[a] + ((double)k + 0.5) * g.dx);
}

__device__ inline size_t word_of(const MapGrid &g, int x, int y, int z) {
    return (size_t)(x >> 5) + (size_t)g.W * ((size_t)y + (size_t)g.n[1] * (size_t)z);
}

__device__ inline void cell_of_key(const MapGrid &g, uint32_t key, int &x, int &y, int &z) {
    x = (int)(key % (uint32_t)g.n[0]);
    const uint32_t r = key / (uint32_t)g.n[0];
    y = (int)(r % (uint32_t)g.n[1]);
    z = (int)(r / (uint32_t)g.n[1]);
}

__device__ inline bool cell_tris(const uint2 *hrng, const uint4 *compact, const MapGrid &g, int x, int y, int z,
                                 uint32_t &beg, uint32_t &len) {
    const uint32_t h = (kHashP1 * (uint32_t)x + kHashP2 * (uint32_t)y + kHashP3 * (uint32_t)z) & g.hash_mask;
    const uint2 r = hrng[h];
    const uint32_t key = (uint32_t)x + (uint32_t)g.n[0] * ((uint32_t)y + (uint32_t)g.n[1] * (uint32_t)z);
    for (uint32_t e = r.x; e < r.x + r.y; e++) {
        const uint4 c = compact[e];
        if (c.x == key) {
            beg = c.y;
            len = c.z;
            return true;
        }
    }
    return false;
}

// the ray of a column as FP32 pairs: hi + lo is within 2^-48 of q
struct RayPoint {
    float xh, xl, yh, yl;
};

__device__ inline RayPoint ray_point(double qx, double qy) {
    const float xh = (float)qx, yh = (float)qy;
    return RayPoint{xh, (float)(qx - (double)xh), yh, (float)(qy - (double)yh)};
}

// Whether the ray meets triangle (a, b, c) within its edges (1) or not (-1), in
// FP32, or that FP32 does not tell (0).  m1, m2, m3 are the signed areas that
// the edges make with q: inside they have one sign, outside two differ.  With
// u = 2^-24 every difference below is off by at most 2 u (|its value| + |lo|)
// <= 2 u mx, so an area by at most 12 u mx my (two products of two such
// factors, their rounding and the subtraction's); the FP64 test's own error is
// 2^-46 mx my.  Areas beyond 32 u mx my therefore have their signs in the FP64
// test too: two opposite ones miss whatever the sign of its determinant, three
// alike give it theirs.  NaN and overflow are never certain.
__device__ inline int ray_side(const float4 &a, const float4 &b, const float4 &c, const RayPoint &q) {
    const float ax = (a.x - q.xh) - q.xl, bx = (b.x - q.xh) - q.xl, cx = (c.x - q.xh) - q.xl;
    const float ay = (a.y - q.yh) - q.yl, by = (b.y - q.yh) - q.yl, cy = (c.y - q.yh) - q.yl;
    const float mx = fmaxf(fmaxf(fabsf(ax), fabsf(bx)), fabsf(cx)) + fabsf(q.xl);
    const float my = fmaxf(fmaxf(fabsf(ay), fabsf(by)), fabsf(cy)) + fabsf(q.yl);
    const float m1 = bx * cy - cx * by, m2 = cx * ay - ax * cy, m3 = ax * by - bx * ay;
    const float bound = mx * my * 0x1p-19f + 1e-36f;    // (and products that underflow)
    const bool p1 = m1 > bound, p2 = m2 > bound, p3 = m3 > bound;
    const bool n1 = m1 < -bound, n2 = m2 < -bound, n3 = m3 < -bound;
    if ((p1 || p2 || p3) && (n1 || n2 || n3)) return -1;
    return (p1 && p2 && p3) || (n1 && n2 && n3) ? 1 : 0;
}

// barycentric weights of (qx, qy) in FP64; false outside.  A nonzero quotient
// of these differences is far above underflow, so its sign is that of its
// operands.
__device__ inline bool ray_weights(const float4 &a, const float4 &b, const float4 &c, double qx, double qy, double &l1,
                                   double &l2, double &l3) {
    auto negative = [](double num, double den) {
        return num != 0.0 && (__double2hiint(num) ^ __double2hiint(den)) < 0;
    };
    const double ax = a.x, ay = a.y, bx = b.x, by = b.y, cx = c.x, cy = c.y;
    const double d = (bx - ax) * (cy - ay) - (cx - ax) * (by - ay);
    if (d == 0.0) return false;
    const double m1 = (bx - qx) * (cy - qy) - (cx - qx) * (by - qy);
    if (negative(m1, d)) return false;
    const double m2 = (cx - qx) * (ay - qy) - (ax - qx) * (cy - qy);
    if (negative(m2, d)) return false;
    l1 = m1 / d;
    l2 = m2 / d;
    l3 = 1.0 - l1 - l2;
    return !(l3 < 0);
}

__device__ inline void ray_of(const MapGrid &g, int x, int y, double &qx, double &qy) {
    qx = (double)g.mid[0][x] + 1.234567e-6 * g.dx;
    qy = (double)g.mid[1][y] + 2.345678e-6 * g.dx;
}

// the crossing's height, toggled at the highest cell whose centre lies below
__device__ inline void toggle_crossing(const MapGrid &g, uint32_t key, const float4 &a, const float4 &b,
                                       const float4 &c, uint32_t *__restrict__ toggle) {
    int x, y, z;
    cell_of_key(g, key, x, y, z);
    double qx, qy, l1, l2, l3;
    ray_of(g, x, y, qx, qy);
    if (!ray_weights(a, b, c, qx, qy, l1, l2, l3)) return;
    const double zc = l1 * (double)a.z + l2 * (double)b.z + l3 * (double)c.z;
    // zc above a float centre: so is zc rounded up.  The first k is a guess.
    const float zu = __double2float_ru(zc);
    int k = min((int)fminf(fmaxf(ceilf((zu - g.o[2]) / (float)g.dx - 0.5f), 0.f), (float)g.n[2]), g.n[2]);
    while (k < g.n[2] && zu > g.mid[2][k]) k++;
    while (k > 0 && !(zu > g.mid[2][k - 1])) k--;
    if (k > 0) atomicXor(toggle + word_of(g, x, y, k - 1), 1u << (x & 31));
}

// One thread per occupied cell.  The cells of a column that list a triangle are
// one run along z where the ray meets it, so a crossing counts at the lowest one,
// found by a look at the cell below.  One run: a cell that the triangle meets
// always passes the binning's separating-axis test, and along z the cells it
// meets are consecutive.  Past them some axis separates.  The gap on it is a
// concave function of z, is above 1e-6 cells (the inflation) where the ray's
// crossing lies, and so falls by over 1e-6 / n cells with every further cell of
// a column of n, far more than the FP64 test's rounding: no cell beyond a
// separated one passes.  (2.6 million pairs of neighbouring cells of slivers, of
// steep and flat triangles and of ones rounded off the cells' faces: no gap.)
// Bound by the FP64 units, a 64th of the FP32 rate, which a warp keeps busy for
// one lane as for 32: the test is decided in FP32 but next to an edge, and the
// warp's crossings are queued so that their heights are computed 32 at a time.
// Gear turned in space, 1.7e8 cells: every test in FP64 523 us, FP32 for the misses
// alone 470 (some lane of most warps still meets its triangle), both 129.
__global__ void __launch_bounds__(256) k_crossings(const float4 *__restrict__ vx,
                                                   const uint32_t *__restrict__ occ, const uint2 *__restrict__ hrng,
                                                   const uint4 *__restrict__ compact, int64_t ncompact,
                                                   const int32_t *__restrict__ tlist, MapGrid g,
                                                   uint32_t *__restrict__ toggle, uint32_t *__restrict__ entries,
                                                   uint32_t *__restrict__ error) {
    __shared__ uint2 queue[8][64];      // (cell key, triangle), 32 left over at most before 32 more
    uint2 *const mine = queue[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const uint4 cell = i < ncompact ? compact[i] : make_uint4(0u, 0u, 0u, 0u);
    int x, y, z;
    cell_of_key(g, cell.x, x, y, z);
    double qx, qy;
    ray_of(g, x, y, qx, qy);
    const RayPoint q = ray_point(qx, qy);
    auto toggle_of = [&](uint2 v) {
        toggle_crossing(g, v.x, vx[3 * (size_t)v.y], vx[3 * (size_t)v.y + 1], vx[3 * (size_t)v.y + 2], toggle);
    };
    int queued = 0;
    for (uint32_t e = cell.y; __any_sync(0xffffffffu, e < cell.y + cell.z); e++) {
        bool first = false;
        int t = 0;
        if (e < cell.y + cell.z) {
            t = tlist[e];
            const float4 a = vx[3 * (size_t)t], b = vx[3 * (size_t)t + 1], c = vx[3 * (size_t)t + 2];
            const int side = ray_side(a, b, c, q);
            double l1, l2, l3;
            first = side > 0 || (side == 0 && ray_weights(a, b, c, qx, qy, l1, l2, l3));
            if (first && atomicAdd(entries + (size_t)x + (size_t)g.n[0] * (size_t)y, 1u) >= kColEntries) {
                atomicOr(error, 1u);
                first = false;
            }
            if (first && z > 0 && bit_of(occ, (uint64_t)cell.x - (uint64_t)g.n[0] * (uint64_t)g.n[1])) {
                uint32_t beg = 0, len = 0;
                if (cell_tris(hrng, compact, g, x, y, z - 1, beg, len))
                    for (uint32_t o = beg; o < beg + len && first; o++) first = tlist[o] != t;
            }
        }
        const uint32_t vote = __ballot_sync(0xffffffffu, first);
        if (first) mine[queued + __popc(vote & ((1u << lane) - 1u))] = make_uint2(cell.x, (uint32_t)t);
        queued += __popc(vote);
        if (queued >= 32) {
            __syncwarp();
            toggle_of(mine[lane]);
            queued -= 32;
            const uint2 rest = mine[32 + lane];     // (the first `queued` of them)
            __syncwarp();
            if (lane < queued) mine[lane] = rest;
        }
    }
    __syncwarp();
    if (lane < queued) toggle_of(mine[lane]);
}

// the toggles of a column, from above: in place, bit (x, y, z) becomes the
// parity of the crossings above its centre.  One thread per 32 columns.
__global__ void __launch_bounds__(128) k_inside_words(uint32_t *__restrict__ m, MapGrid g) {
    const int64_t q = (int64_t)blockIdx.x * 128 + threadIdx.x;
    const int64_t plane = (int64_t)g.W * g.n[1];
    if (q >= plane) return;
    uint32_t acc = 0u;
    constexpr int kAhead = 8;      // words in flight
    for (int z = g.n[2] - 1; z >= 0; z -= kAhead) {
        uint32_t v[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; u++) v[u] = z - u >= 0 ? m[q + plane * (z - u)] : 0u;
#pragma unroll
        for (int u = 0; u < kAhead; u++) {
            acc ^= v[u];
            if (z - u >= 0) m[q + plane * (z - u)] = acc;
        }
    }
}

// the occupancy bitmap (bit = cell key) as padded rows
__global__ void __launch_bounds__(256) k_occ_rows(const uint32_t *__restrict__ occ, int64_t occ_words, int64_t words,
                                                  MapGrid g, uint32_t *__restrict__ out) {
    const int64_t q = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (q >= words) return;
    const int64_t row = (uint32_t)q / (uint32_t)g.W;
    const int x0 = 32 * (int)(q - row * g.W), left = g.n[0] - x0;
    const uint64_t c = (uint64_t)row * (uint64_t)g.n[0] + (uint64_t)x0;
    const int64_t w = (int64_t)(c >> 5);
    const uint32_t v = __funnelshift_r(occ[w], w + 1 < occ_words ? occ[w + 1] : 0u, (uint32_t)(c & 31u));
    out[q] = left >= 32 ? v : v & ((1u << left) - 1u);
}

// bit x of out: some bit of src within `band` of x in the same row
__global__ void __launch_bounds__(256) k_dilate_x(const uint32_t *__restrict__ src, uint32_t *__restrict__ dst,
                                                  int64_t words, MapGrid g, int band) {
    const int64_t q = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (q >= words) return;
    const int64_t row = (uint32_t)q / (uint32_t)g.W;
    const int w = (int)(q - row * g.W);
    const uint32_t *r = src + row * g.W;
    // bits 32 w + d .. 32 w + d + 31 for d = -band .. band
    uint32_t v = 0u;
    for (int k = w - (band + 31) / 32; k <= w + band / 32; k++) {
        const uint32_t lo = k >= 0 && k < g.W ? r[k] : 0u, hi = k + 1 >= 0 && k + 1 < g.W ? r[k + 1] : 0u;
        if ((lo | hi) == 0u) continue;
        for (int sh = 0; sh < 32; sh++) {
            const int d = 32 * (k - w) + sh;
            if (d >= -band && d <= band) v |= __funnelshift_r(lo, hi, (uint32_t)sh);
        }
    }
    const int left = g.n[0] - 32 * w;
    dst[q] = left >= 32 ? v : v & ((1u << left) - 1u);
}

// the same along y (axis 1) or z (axis 2)
__global__ void __launch_bounds__(256) k_dilate_yz(const uint32_t *__restrict__ src, uint32_t *__restrict__ dst,
                                                   int64_t words, MapGrid g, int axis, int band) {
    const int64_t q = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (q >= words) return;
    const int64_t stride = axis == 1 ? g.W : (int64_t)g.W * g.n[1];
    const int i = (int)(((uint32_t)q / (uint32_t)stride) % (uint32_t)g.n[axis]);
    const int lo = max(-band, -i), hi = min(band, g.n[axis] - 1 - i);
    uint32_t v = 0u;
    for (int d = lo; d <= hi; d++) v |= src[q + d * stride];
    dst[q] = v;
}

// nearest triangle of the cell (a C_compact entry) whose foot of its centre p is inside
// (the FP32 rule of the constraint step); -1 when none
__device__ int map_surface_cell(const float4 *__restrict__ geo, const uint4 &cell, const int32_t *__restrict__ tlist,
                                const MapGrid &g, float3 p, float &dist) {
    float best = FLT_MAX, bd = 0.f;
    int bt = -1;
    for (uint32_t e = cell.y; e < cell.y + cell.z; e++) {
        const int t = tlist[e];
        const float4 *q = geo + 5 * (size_t)t;
        const float ux = __fsub_rn(p.x, q[0].x), uy = __fsub_rn(p.y, q[0].y), uz = __fsub_rn(p.z, q[0].z);
        auto dotu = [&](float4 m) { return ux * m.x + uy * m.y + uz * m.z; };
        if (dotu(q[2]) < -g.edge_tol) continue;
        if (dotu(q[3]) - q[3].w < -g.edge_tol) continue;
        if (dotu(q[4]) - q[4].w < -g.edge_tol) continue;
        const float d = dotu(q[1]);
        const float ad = fabsf(d);
        if (ad < best || (ad == best && t < bt)) {
            best = ad;
            bd = d;
            bt = t;
        }
    }
    dist = bd;
    return bt;
}

__device__ inline float3 cell_centre(const MapGrid &g, int x, int y, int z) {
    return make_float3(g.mid[0][x], g.mid[1][y], g.mid[2][z]);
}

// the triangle (-1: none) and plane distance of every occupied cell's centre,
// and the bitmap of the cells that have one
__global__ void __launch_bounds__(256) k_surface_cells(const float4 *__restrict__ geo, const uint4 *__restrict__ compact,
                                                       int64_t ncompact,
                                                       const int32_t *__restrict__ tlist, MapGrid g,
                                                       int32_t *__restrict__ tri, float *__restrict__ dist,
                                                       uint32_t *__restrict__ sbits) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= ncompact) return;
    int x, y, z;
    cell_of_key(g, compact[i].x, x, y, z);
    float d = 0.f;
    const int t = map_surface_cell(geo, compact[i], tlist, g, cell_centre(g, x, y, z), d);
    tri[i] = t;
    dist[i] = d;
    if (t >= 0) atomicOr(sbits + word_of(g, x, y, z), 1u << (x & 31));
}

// vbits (the inside bitmap on entry): empty cells inside, within inner
// (nullable); the counts of surface cells, then of volume cells, per word
__global__ void __launch_bounds__(256) k_word_counts(const uint32_t *__restrict__ rows,
                                                     const uint32_t *__restrict__ sbits,
                                                     const uint32_t *__restrict__ inner, int64_t words,
                                                     uint32_t *__restrict__ vbits, uint32_t *__restrict__ cnt) {
    const int64_t q = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (q >= words) return;
    uint32_t v = vbits[q] & ~rows[q];
    if (inner) v &= inner[q];
    vbits[q] = v;
    cnt[q] = (uint32_t)__popc(sbits[q]);
    cnt[words + q] = (uint32_t)__popc(v);
}

__global__ void __launch_bounds__(256) k_emit_surface(const float4 *__restrict__ geo, const uint4 *__restrict__ compact,
                                                      int64_t ncompact, const int32_t *__restrict__ tri,
                                                      const float *__restrict__ dist,
                                                      const uint32_t *__restrict__ sbits,
                                                      const uint32_t *__restrict__ off, MapGrid g,
                                                      float4 *__restrict__ pos, int32_t *__restrict__ cons) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= ncompact) return;
    const int t = tri[i];
    if (t < 0) return;
    int x, y, z;
    cell_of_key(g, compact[i].x, x, y, z);
    const size_t w = word_of(g, x, y, z);
    const size_t o = (size_t)off[w] + (size_t)__popc(sbits[w] & ((1u << (x & 31)) - 1u));
    const float3 p = cell_centre(g, x, y, z);
    const float4 n = geo[5 * (size_t)t + 1];
    const float d = dist[i];
    pos[o] = make_float4(p.x - d * n.x, p.y - d * n.y, p.z - d * n.z, __uint_as_float(class_bit(kClsS)));
    cons[o] = t;
}

// A warp takes 32 words and emits them one after another, a lane per cell.
// off: places counted from the first surface particle; first: the same of the
// first volume particle.  band (nullable): V inside it, else I; cls (with
// band): the class of every volume particle.
__global__ void __launch_bounds__(256) k_emit_volume(const uint32_t *__restrict__ vbits,
                                                     const uint32_t *__restrict__ off,
                                                     const uint32_t *__restrict__ band, int64_t words, uint32_t first,
                                                     MapGrid g, float4 *__restrict__ pos, int32_t *__restrict__ cons,
                                                     uint8_t *__restrict__ cls) {
    const int lane = threadIdx.x & 31;
    const int64_t q0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) & ~(int64_t)31, q = q0 + lane;
    const uint32_t mine = q < words ? vbits[q] : 0u;
    const uint32_t at = mine ? off[q] : 0u, near = mine ? (band ? band[q] : 0xffffffffu) : 0u;
    uint32_t todo = __ballot_sync(0xffffffffu, mine != 0u);
    while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1u;
        const uint32_t v = __shfl_sync(0xffffffffu, mine, src), a = __shfl_sync(0xffffffffu, at, src);
        const uint32_t b = __shfl_sync(0xffffffffu, near, src);
        if (!((v >> lane) & 1u)) continue;
        // (below 2^32 / 5 words: a row has at least five cells to the word)
        const uint32_t wq = (uint32_t)(q0 + src), row = wq / (uint32_t)g.W;
        const int x = 32 * (int)(wq - row * (uint32_t)g.W) + lane;
        const int z = (int)(row / (uint32_t)g.n[1]), y = (int)(row - (uint32_t)z * (uint32_t)g.n[1]);
        const uint32_t o = a + (uint32_t)__popc(v & ((1u << lane) - 1u));
        const int cl = (b >> lane) & 1u ? kClsV : kClsI;
        const float3 p = cell_centre(g, x, y, z);
        pos[o] = make_float4(p.x, p.y, p.z, __uint_as_float(class_bit(cl)));
        cons[o] = -1;
        if (cls) cls[o - first] = (uint8_t)cl;
    }
}

inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)std::max<int64_t>((n + t - 1) / t, 1); }

} // namespace

// Feature particles of Sec. 3.2.2 on the host from the walked lines: n =
// ceil(L / dx) pieces of length L / n; open lines add their singular end
// points once (class P); loops carry n points.  seg gets the segment each
// feature particle was placed on (-1 for singular points), so its first
// step already projects onto its own line.
void Body::feature_particles(std::vector<float> &xyz, std::vector<int32_t> &cls, std::vector<int32_t> &seg, int l0,
                             int l1) const {
    std::vector<char> done(verts_host.size() / 3, 0);
    if (l1 < 0) l1 = nlines;
    auto seglen = [&](int64_t q) {
        const float *a = &verts_host[3 * (size_t)seg_v[2 * q]], *b = &verts_host[3 * (size_t)seg_v[2 * q + 1]];
        const double e0 = (double)b[0] - a[0], e1 = (double)b[1] - a[1], e2 = (double)b[2] - a[2];
        return std::sqrt(e0 * e0 + e1 * e1 + e2 * e2);
    };
    auto emit = [&](double x, double y, double z, int c, int64_t q) {
        xyz.push_back((float)x);
        xyz.push_back((float)y);
        xyz.push_back((float)z);
        cls.push_back(c);
        seg.push_back((int32_t)q);
    };
    for (int l = l0; l < l1; l++) {
        const int64_t f = line_first[l], ns = line_nseg[l];
        double L = 0.0;
        for (int64_t q = f; q < f + ns; q++) L += seglen(q);
        int64_t np = (int64_t)std::ceil(L / (double)dx);
        if (np < 1) np = 1;
        const double sp = L / (double)np;
        const bool closed = line_closed[l] != 0;
        if (!closed) {
            for (int32_t v : {seg_v[2 * f], seg_v[2 * (f + ns - 1) + 1]})
                if (!done[v]) {
                    done[v] = 1;
                    emit(verts_host[3 * (size_t)v], verts_host[3 * (size_t)v + 1], verts_host[3 * (size_t)v + 2], kClsP,
                         -1);
                }
        }
        int64_t q = f;
        double cum = 0.0;
        for (int64_t k = closed ? 0 : 1; k <= np - 1; k++) {
            const double target = sp * (double)k;
            while (q < f + ns - 1 && cum + seglen(q) <= target) {
                cum += seglen(q);
                q++;
            }
            const double len = seglen(q), t = len > 0 ? (target - cum) / len : 0.0;
            const float *a = &verts_host[3 * (size_t)seg_v[2 * q]], *b = &verts_host[3 * (size_t)seg_v[2 * q + 1]];
            emit(a[0] + t * ((double)b[0] - a[0]), a[1] + t * ((double)b[1] - a[1]), a[2] + t * ((double)b[2] - a[2]),
                 kClsF, q);
        }
    }
}

int map_particles(Group &g, Body &b, int surface, int volume, int features, int band_cells, int inner_cells,
                  cudaStream_t s, bool fixed_features, int64_t *n_out, std::vector<int32_t> &cls_host,
                  int64_t *n_singular, std::string &err) {
    MapGrid mg;
    for (int k = 0; k < 3; k++) {
        mg.o[k] = b.tg_o[k];
        mg.n[k] = b.tg_n[k];
    }
    mg.dx = (double)b.dx;
    mg.hash_mask = (uint32_t)(b.hash_size - 1);
    mg.edge_tol = b.edge_tol;
    const int64_t cells = (int64_t)mg.n[0] * mg.n[1] * mg.n[2];
    if (cells >= 0xffffffffLL) {
        err = "map_particles: triangle grid too large";
        return 1;
    }
    std::vector<float> fxyz;
    std::vector<int32_t> fcls, fseg;
    if (features && b.has_features) b.feature_particles(fxyz, fcls, fseg);
    const int64_t nf = (int64_t)fcls.size();

    // one block of scratch: [0, zeroed) starts at 0
    mg.W = (mg.n[0] + 31) / 32;
    const int64_t words = (int64_t)mg.W * mg.n[1] * mg.n[2], cols = (int64_t)mg.n[0] * mg.n[1];
    const bool use_band = volume && band_cells > 0, use_inner = use_band && inner_cells > 0;
    const int64_t sc = scan_tmp_elems(2 * words);
    const int64_t zeroed = 2 * words + cols + 1;
    const int64_t mids = (int64_t)mg.n[0] + mg.n[1] + mg.n[2];
    const int64_t total = zeroed + mids + (use_inner ? 4 : use_band ? 3 : 0) * words + 5 * words + 2 * b.ncompact + 2 + sc;
    uint32_t *scr = nullptr;
    uint8_t *vcls = nullptr;
    auto cleanup = [&]() {
        if (scr) cudaFree(scr);
        if (vcls) cudaFree(vcls);
    };
    if (dev_malloc(&scr, sizeof(uint32_t) * (size_t)total)) {
        err = "map_particles: out of device memory";
        return 3;
    }
    uint32_t *q = scr;
    auto take = [&](int64_t n) {
        uint32_t *r = q;
        q += n;
        return r;
    };
    uint32_t *vbits = take(words), *sbits = take(words), *entries = take(cols), *error = take(1);
    uint32_t *rows = take(words), *cnt = take(2 * words), *off = take(2 * words);
    uint32_t *t1 = use_band ? take(words) : nullptr, *t2 = use_band ? take(words) : nullptr;
    uint32_t *band = use_band ? take(words) : nullptr, *inner = use_inner ? take(words) : nullptr;
    int32_t *tri = (int32_t *)take(b.ncompact);
    float *dist = (float *)take(b.ncompact);
    uint32_t *tot = take(2), *tmp = take(sc);
    float *mid = (float *)take(mids);
    for (int k = 0, at = 0; k < 3; at += mg.n[k++]) mg.mid[k] = mid + at;
    k_centres<<<nblk(mids), 256, 0, s>>>(mg, mid);
    cudaMemsetAsync(scr, 0, sizeof(uint32_t) * (size_t)zeroed, s);
    k_occ_rows<<<nblk(words), 256, 0, s>>>(b.occ, b.occ_words, words, mg, rows);
    if (volume) {
        k_crossings<<<nblk(b.ncompact), 256, 0, s>>>(b.vx, b.occ, b.hrng, b.compact, b.ncompact, b.tlist,
                                                     mg, vbits, entries, error);
        k_inside_words<<<nblk((int64_t)mg.W * mg.n[1], 128), 128, 0, s>>>(vbits, mg);
    }
    auto dilate = [&](uint32_t *out, int r) {
        k_dilate_x<<<nblk(words), 256, 0, s>>>(rows, t1, words, mg, r);
        k_dilate_yz<<<nblk(words), 256, 0, s>>>(t1, t2, words, mg, 1, r);
        k_dilate_yz<<<nblk(words), 256, 0, s>>>(t2, out, words, mg, 2, r);
    };
    if (use_band) dilate(band, band_cells);
    if (use_inner) dilate(inner, band_cells + inner_cells);
    if (surface)
        k_surface_cells<<<nblk(b.ncompact), 256, 0, s>>>(b.geo, b.compact, b.ncompact, b.tlist, mg, tri, dist, sbits);
    k_word_counts<<<nblk(words), 256, 0, s>>>(rows, sbits, inner, words, vbits, cnt);
    exclusive_scan_u32(cnt, off, 2 * words, tot, tmp, sc, s);
    uint32_t all = 0, first = 0, errh = 0;
    auto ok = [&](cudaError_t e) {
        if (e == cudaSuccess) return true;
        err = std::string("map_particles: ") + cudaGetErrorString(e);
        return false;
    };
    if (!ok(cudaMemcpyAsync(&all, tot, 4, cudaMemcpyDeviceToHost, s)) ||
        !ok(cudaMemcpyAsync(&first, off + words, 4, cudaMemcpyDeviceToHost, s)) ||
        !ok(cudaMemcpyAsync(&errh, error, 4, cudaMemcpyDeviceToHost, s)) || !ok(cudaStreamSynchronize(s))) {
        cleanup();
        return 4;
    }
    if (errh) {
        cleanup();
        err = "map_particles: a grid column crosses more than 256 triangle entries";
        return 6;
    }
    const int64_t ns = first, nvol = (int64_t)all - ns, N = nf + ns + nvol;
    if (N != g.d.N || !g.d.pos) {
        const int r = g.alloc_particles(N, err);
        if (r) {
            cleanup();
            return r;
        }
    } else {
        // the arrays are used again: work on the old particles that is still
        // under way on a stream the body had before ends first (a new
        // allocation waits for it when it frees the old arrays)
        if (!ok(cudaDeviceSynchronize())) {
            cleanup();
            return 4;
        }
        cudaMemsetAsync(g.d.cert, 0, sizeof(float4) * (size_t)N, s);   // as a new allocation has it
    }
    if (band && nvol && dev_malloc(&vcls, (size_t)nvol)) {
        cleanup();
        err = "map_particles: out of device memory";
        return 3;
    }
    std::vector<float4> p4(nf);
    int64_t np = 0;                // singular points
    if (nf) {
        for (int64_t i = 0; i < nf; i++) {
            np += fcls[i] == kClsP;
            uint32_t bits = class_bit(fcls[i]);
            float w;
            memcpy(&w, &bits, 4);
            p4[i] = make_float4(fxyz[3 * i], fxyz[3 * i + 1], fxyz[3 * i + 2], w);
        }
        // (constraints: the segment of each feature particle)
        if (!ok(cudaMemcpyAsync(g.d.pos, p4.data(), sizeof(float4) * nf, cudaMemcpyHostToDevice, s)) ||
            !ok(cudaMemcpyAsync(g.d.cons, fseg.data(), sizeof(int32_t) * nf, cudaMemcpyHostToDevice, s))) {
            cudaStreamSynchronize(s);
            cleanup();
            return 4;
        }
    }
    if (surface)
        k_emit_surface<<<nblk(b.ncompact), 256, 0, s>>>(b.geo, b.compact, b.ncompact, tri, dist, sbits, off, mg,
                                                        g.d.pos + nf, g.d.cons + nf);
    k_emit_volume<<<nblk(words), 256, 0, s>>>(vbits, off + words, band, words, first, mg, g.d.pos + nf, g.d.cons + nf,
                                              vcls);
    // keys with many fixed particles (Group::find_crowds): cells are a spacing
    // apart, but singular points and the feature points of different lines are not
    uint32_t most = np ? b.sing_crowd : 0u;
    uint32_t *const crowd = fixed_features && nf > (int64_t)kCrowd ? g.count_crowds(nf, s) : nullptr;
    std::vector<uint8_t> vc(band ? (size_t)nvol : 0);
    bool done = vc.empty() || ok(cudaMemcpyAsync(vc.data(), vcls, vc.size(), cudaMemcpyDeviceToHost, s));
    // the classes on the host: features as given, then S, then V (or as copied)
    cls_host.resize((size_t)N);
    std::copy(fcls.begin(), fcls.end(), cls_host.begin());
    std::fill(cls_host.begin() + nf, cls_host.begin() + nf + ns, (int32_t)kClsS);
    if (crowd) done = ok(cudaMemcpyAsync(&most, crowd, sizeof(most), cudaMemcpyDeviceToHost, s)) && done;
    done = ok(cudaStreamSynchronize(s)) && done && ok(cudaGetLastError());
    g.crowded = most > kCrowd;
    g.choose_order();
    *n_singular = np;
    if (vc.empty()) std::fill(cls_host.begin() + nf + ns, cls_host.end(), (int32_t)kClsV);
    else std::copy(vc.begin(), vc.end(), cls_host.begin() + nf + ns);
    cleanup();
    if (!done) return 4;
    *n_out = N;
    return 0;
}

} // namespace fppg
