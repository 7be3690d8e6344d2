// Uniformity statistics (fppg_stats): the kernel sum rho of every S, V and F
// particle, its mean and standard deviation per class, the smallest masked
// pair distance.
//
//   k_density      rho in key order, and per block the class sums and counts
//                  in FP64 and the smallest r^2
//   k_stat_sums    one block adds the blocks' shares up: counts and means
//   k_deviation    per block the class sums of (rho - mean)^2
//   k_stat_sums    the same for the deviations
// Every sum is a fixed tree (no atomics: the same bits on every run), and the
// means stay on the device, so the host waits once.
#include <cfloat>
#include <cmath>

#include "body.h"
#include "pairs.cuh"

namespace fppg {

namespace {

constexpr int TPB = 256;
inline unsigned nblocks(int64_t n) { return (unsigned)std::max<int64_t>((n + TPB - 1) / TPB, 1); }

// classes that are counted (S, V, F), and the values a block leaves: sums,
// counts, the smallest r^2
constexpr int kStatClasses = 3;
constexpr int kShare = 2 * kStatClasses + 1;

__device__ inline double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// the sum of v over the block's threads of class c, for c = 0..2, in thread
// 0's out[]; sh: 8 x 3 doubles.  Warps without the class add nothing.
__device__ inline void block_class_sums(double v, int cls, double (*sh)[kStatClasses], double *out) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < kStatClasses; c++) {
        double t = 0.0;
        if (__any_sync(0xffffffffu, cls == c)) t = warp_sum(cls == c ? v : 0.0);
        if (lane == 0) sh[w][c] = t;
    }
    __syncthreads();
    if (threadIdx.x < kStatClasses) {
        double t = 0.0;
        for (int q = 0; q < TPB / 32; q++) t += sh[q][threadIdx.x];
        out[threadIdx.x] = t;
    }
}

// Walks the slots that the reach cut keeps, two at a time (as the energy
// does), where the sums took the whole 27 cells one by one: 540 k particles
// 302 -> 154 us, bound like the force pass by the pair arithmetic.  (The sums
// that follow took 1,915 us as one FP64 atomic per particle on three
// addresses; block shares take 13 + 2 x 6 us.)  The particle itself adds exactly 1 to the kernel
// sum; the smallest distance is taken over r^2 < (2h)^2 in FP32 without
// contraction, itself excluded.
__global__ void __launch_bounds__(TPB) k_density(const float4 *__restrict__ pos_s, const float4 *__restrict__ pos_p,
                                                 int64_t N, const AsmParams *__restrict__ P,
                                                 const uint32_t *__restrict__ fstart, float *__restrict__ rho_s,
                                                 double *__restrict__ part) {
    __shared__ double sh[TPB / 32][kStatClasses], out[kStatClasses];
    __shared__ int s_cnt[TPB / 32][kStatClasses];
    __shared__ float s_min[TPB / 32];
    const int64_t k = (int64_t)blockIdx.x * TPB + threadIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const float4 p = k < N ? pos_s[k] : make_float4(0.f, 0.f, 0.f, 0.f);
    const AsmParams &A = P[k < N ? body_of(p.w) : 0];
    int cls = k < N ? cls_of(p.w) : kClsP;
    if (k < N && is_ghost(p.w)) cls = kClsP;             // not counted
    const bool on = cls <= kClsF, mob = on && is_mobile(cls, A);
    const uint32_t mbits = on ? acts_on_bits(cls) : 0u;
    const float hih = A.half_inv_h, R2 = A.R2;
    const float2 npx = make_float2(-p.x, -p.x), npy = make_float2(-p.y, -p.y), npz = make_float2(-p.z, -p.z);
    const float4 *pos_b = pos_p + (N + 1) / 2;
    float2 acc = make_float2(0.f, 0.f);
    float rmin = FLT_MAX;
    for_row_ranges(p, on, A, fstart, [&](uint32_t s, uint32_t e) {
        for_pairs(s, e, [&](auto edge, uint32_t m) {
            constexpr bool EDGE = decltype(edge)::value;
            const PairGeo g = pair_geo(pos_p, pos_b, m, npx, npy, npz, hih);
            const float2 t2 = __fmul2_rn(g.t, g.t);
            const float2 poly = __ffma2_rn(g.r, make_float2(4.f * hih, 4.f * hih), make_float2(1.f, 1.f));
            const float2 wt = __fmul2_rn(__fmul2_rn(t2, t2), poly);
            const bool k0 = (!EDGE || 2 * m >= s) && (mbits & g.w0) != 0u;
            const bool k1 = (!EDGE || 2 * m + 1 < e) && (mbits & g.w1) != 0u;
            acc = __fadd2_rn(acc, make_float2(k0 ? wt.x : 0.f, k1 ? wt.y : 0.f));
            if (k0 && 2 * m != (uint32_t)k && g.r2.x < R2) rmin = fminf(rmin, g.r2.x);
            if (k1 && 2 * m + 1 != (uint32_t)k && g.r2.y < R2) rmin = fminf(rmin, g.r2.y);
        });
    });
    // a class that acts on its own always meets itself above
    const float rho = A.alpha * (acc.x + acc.y);
    if (k < N) rho_s[k] = rho;
    if (!mob) rmin = FLT_MAX;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rmin = fminf(rmin, __shfl_xor_sync(0xffffffffu, rmin, o));
    if (lane == 0) s_min[w] = rmin;
#pragma unroll
    for (int c = 0; c < kStatClasses; c++) {
        const int n = __popc(__ballot_sync(0xffffffffu, cls == c));
        if (lane == 0) s_cnt[w][c] = n;
    }
    block_class_sums((double)rho, cls, sh, out);
    __syncthreads();
    double *o = part + (size_t)blockIdx.x * kShare;
    if (threadIdx.x < kStatClasses) {
        int n = 0;
        for (int q = 0; q < TPB / 32; q++) n += s_cnt[q][threadIdx.x];
        o[threadIdx.x] = out[threadIdx.x];
        o[kStatClasses + threadIdx.x] = (double)n;
    }
    if (threadIdx.x == 0) {
        float m = s_min[0];
        for (int q = 1; q < TPB / 32; q++) m = fminf(m, s_min[q]);
        o[2 * kStatClasses] = (double)m;
    }
}

__global__ void __launch_bounds__(TPB) k_deviation(const float4 *__restrict__ pos_s, const float *__restrict__ rho_s,
                                                   int64_t N, const double *__restrict__ mean,
                                                   double *__restrict__ part) {
    __shared__ double sh[TPB / 32][kStatClasses], out[kStatClasses];
    const int64_t k = (int64_t)blockIdx.x * TPB + threadIdx.x;
    const float w = k < N ? pos_s[k].w : 0.f;
    int cls = k < N ? cls_of(w) : kClsP;
    if (k < N && is_ghost(w)) cls = kClsP;
    double d = 0.0;
    if (cls <= kClsF) d = (double)rho_s[k] - mean[cls];
    block_class_sums(d * d, cls, sh, out);
    __syncthreads();
    if (threadIdx.x < kStatClasses) part[(size_t)blockIdx.x * kShare + threadIdx.x] = out[threadIdx.x];
}

// one block: the shares of nb blocks added up, four warps to a value.  FIRST:
// res[0..2] the means, res[3..5] the counts, res[6] the smallest r^2; else
// res[7..9] the sums of squares.
template <bool FIRST>
__global__ void __launch_bounds__(32 * 4 * kShare) k_stat_sums(const double *__restrict__ part, int64_t nb,
                                                               double *__restrict__ res) {
    __shared__ double sh[kShare][4];
    const int lane = threadIdx.x & 31, c = (threadIdx.x >> 5) % kShare, q = (threadIdx.x >> 5) / kShare;
    const bool low = c == 2 * kStatClasses;      // a minimum, not a sum
    double v = low ? (double)FLT_MAX : 0.0;
    if (FIRST || c < kStatClasses) {
#pragma unroll 4
        for (int64_t b = 32 * q + lane; b < nb; b += 128) {
            const double t = part[b * kShare + c];
            v = low ? fmin(v, t) : v + t;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double t = __shfl_xor_sync(0xffffffffu, v, o);
            v = low ? fmin(v, t) : v + t;
        }
        if (lane == 0) sh[c][q] = v;
    }
    __syncthreads();
    if (threadIdx.x >= kShare || (!FIRST && threadIdx.x >= kStatClasses)) return;
    const int k = threadIdx.x;
    const double *x = sh[k];
    if (!FIRST) {
        res[kShare + k] = (x[0] + x[1]) + (x[2] + x[3]);
    } else if (k < kStatClasses) {
        const double *n = sh[kStatClasses + k];
        const double cnt = (n[0] + n[1]) + (n[2] + n[3]);
        res[k] = cnt > 0.0 ? ((x[0] + x[1]) + (x[2] + x[3])) / cnt : 0.0;
    } else {
        res[k] = k == 2 * kStatClasses ? fmin(fmin(x[0], x[1]), fmin(x[2], x[3])) : (x[0] + x[1]) + (x[2] + x[3]);
    }
}

} // namespace

// doubles of scratch for N particles: every block's share, then the results
int64_t stat_scratch(int64_t n) { return (int64_t)nblocks(n) * kShare + kShare + kStatClasses; }

int stats(Group &g, cudaStream_t s, double *mean, double *sd, double *minpair, double *maxdisp, int64_t *cnt,
          std::string &err) {
    DevGroup &d = g.d;
    double h[kShare + kStatClasses] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, (double)FLT_MAX, 0.0, 0.0, 0.0};
    uint32_t md = 0;
    cudaMemcpyAsync(&md, d.maxdisp, 4, cudaMemcpyDeviceToHost, s);   // (the grid build resets it)
    if (d.N > 0) {
        const int64_t nb = nblocks(d.N);
        double *res = d.stat + nb * kShare;
        float *rho = d.coef_s;
        build_grid(g, s);
        k_density<<<(unsigned)nb, TPB, 0, s>>>(d.pos_s, d.pos_p, d.N, d.params, d.fstart, rho, d.stat);
        k_stat_sums<true><<<1, 32 * 4 * kShare, 0, s>>>(d.stat, nb, res);
        k_deviation<<<(unsigned)nb, TPB, 0, s>>>(d.pos_s, rho, d.N, res, d.stat);
        k_stat_sums<false><<<1, 32 * 4 * kShare, 0, s>>>(d.stat, nb, res);
        cudaMemcpyAsync(h, res, sizeof(h), cudaMemcpyDeviceToHost, s);
    }
    cudaError_t e = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = cudaGetLastError();
    for (int c = 0; c < kStatClasses; c++) {
        mean[c] = h[c];
        cnt[c] = (int64_t)h[kStatClasses + c];
        sd[c] = cnt[c] > 0 ? std::sqrt(h[kShare + c] / (double)cnt[c]) : 0.0;
    }
    float mdf;
    memcpy(&mdf, &md, 4);
    const float dx = g.hp[0].dx;
    const float r2 = (float)h[2 * kStatClasses];
    *minpair = r2 >= FLT_MAX ? INFINITY : (double)std::sqrt(r2) / dx;
    *maxdisp = (double)mdf / dx;
    if (e != cudaSuccess) {
        err = std::string("stats: ") + cudaGetErrorString(e);
        return 4;
    }
    return 0;
}

} // namespace fppg
