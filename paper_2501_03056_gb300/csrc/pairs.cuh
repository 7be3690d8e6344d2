// The pair walk shared by the energy and the statistics.
#pragma once

#include <type_traits>

#include "fppg_internal.cuh"

namespace fppg {

// The pair sums walk the same candidates as the force pass: per grid row of
// the 3 x 3 rows around p, the slots that the reach cut keeps (a superset of
// the particles within 2h), read two at a time from the slot-pair copy
// ({x0, x1, y0, y1}, {z0, z1, w0, w1}) into packed FP32x2 operands.  The
// first and last pair of a range may hold a slot outside it (EDGE), masked
// out.  Weights use max(1 - r / 2h, 0), so a slot beyond 2h adds exactly 0
// and one within rounding of 2h a term below 1e-18 of the largest.
template <typename F>
__device__ inline void for_row_ranges(const float4 &p, bool on, const AsmParams &A, const uint32_t *fstart, F &&f) {
    const int ny = A.ng_n[1], nz = A.ng_n[2];
    const GridPoint g = grid_point(A, p.x, p.y, p.z);
    const int cy = g.c[1], cz = g.c[2];
    for (int dz = -1; dz <= 1; dz++) {
        const int z = cz + dz;
        const float gz = row_gap(g.t[2], cz, dz, g.slack);
        for (int dy = -1; dy <= 1; dy++) {
            const int y = cy + dy;
            uint32_t s = 0xffffffffu, e = 0u;
            if (on && z >= 0 && z < nz && y >= 0 && y < ny) {
                const uint32_t row = A.key_base + (uint32_t)A.ng_n[0] * grid_row(A, y, z);
                row_slots(A, fstart, g, row_gap(g.t[1], cy, dy, g.slack), gz, row, s, e);
            }
            f(s, e);
        }
    }
}

// the slot pairs [s >> 1, (e + 1) >> 1) of range [s, e): f(edge, m) with
// edge true for the first and the last
template <typename F>
__device__ inline void for_pairs(uint32_t s, uint32_t e, F &&f) {
    if (s >= e) return;
    uint32_t m = s >> 1;
    const uint32_t m1 = (e + 1) >> 1;
    f(std::true_type{}, m);
    if (m + 1 >= m1) return;
    for (m = m + 1; m + 1 < m1; m++) f(std::false_type{}, m);
    f(std::true_type{}, m1 - 1);
}

struct PairGeo {
    float2 dx, dy, dz, t;   // q - p per axis; max(1 - r / 2h, 0)
    float2 r, r2;
    uint32_t w0, w1;        // class bits of the two slots
};

// pos_p: the {x, y} halves of the slot pairs, pos_b: the {z, w} halves
__device__ inline PairGeo pair_geo(const float4 *__restrict__ pos_p, const float4 *__restrict__ pos_b, uint32_t m,
                                   float2 npx, float2 npy, float2 npz, float hih) {
    const float4 A = pos_p[m], B = pos_b[m];
    PairGeo o;
    o.dx = __fadd2_rn(make_float2(A.x, A.y), npx);
    o.dy = __fadd2_rn(make_float2(A.z, A.w), npy);
    o.dz = __fadd2_rn(make_float2(B.x, B.y), npz);
    o.r2 = __fadd2_rn(__fadd2_rn(__fmul2_rn(o.dx, o.dx), __fmul2_rn(o.dy, o.dy)), __fmul2_rn(o.dz, o.dz));
    o.r = make_float2(sqrt_approx(o.r2.x), sqrt_approx(o.r2.y));
    const float2 t = __ffma2_rn(o.r, make_float2(-hih, -hih), make_float2(1.f, 1.f));
    o.t = make_float2(fmaxf(t.x, 0.f), fmaxf(t.y, 0.f));
    o.w0 = __float_as_uint(B.z);
    o.w1 = __float_as_uint(B.w);
    return o;
}

// The same for sums that take no decision on r^2: fused multiply-adds and the
// weight max(1 - r / 2h, 0) from a saturating FMA.  CLS: the class bits are
// wanted; else only {z, z'} of the second half is read (24 bytes a pair
// instead of 32).
template <bool CLS>
__device__ inline PairGeo pair_sum_geo(const float4 *__restrict__ pos_p, const float4 *__restrict__ pos_b, uint32_t m,
                                       float2 npx, float2 npy, float2 npz, float hih) {
    const float4 A = pos_p[m];
    PairGeo o;
    float2 z;
    if (CLS) {
        const float4 B = pos_b[m];
        z = make_float2(B.x, B.y);
        o.w0 = __float_as_uint(B.z);
        o.w1 = __float_as_uint(B.w);
    } else {
        z = *reinterpret_cast<const float2 *>(pos_b + m);
        o.w0 = o.w1 = 0u;
    }
    o.dx = __fadd2_rn(make_float2(A.x, A.y), npx);
    o.dy = __fadd2_rn(make_float2(A.z, A.w), npy);
    o.dz = __fadd2_rn(z, npz);
    o.r2 = __ffma2_rn(o.dz, o.dz, __ffma2_rn(o.dy, o.dy, __fmul2_rn(o.dx, o.dx)));
    o.r = make_float2(sqrt_approx(o.r2.x), sqrt_approx(o.r2.y));
    o.t = make_float2(__saturatef(fmaf(o.r.x, -hih, 1.f)), __saturatef(fmaf(o.r.y, -hih, 1.f)));
    return o;
}

} // namespace fppg
