// The relaxation hot path (Algorithm 1, Sec. 3.3) for a group of bodies.
//
// Per iteration, all bodies at once:
//   grid build  A1-A3  cell key per particle (FP32 rule, no contraction), the
//                      order by (key, id), positions and constraint ids in
//                      that order, the dense table of the first slot of
//                      every fine key: a counting sort (k_keys_count ..
//                      k_rank_gather), or k_keys, a stable radix sort,
//                      k_gather and the table from the sorted keys
//   k_force         A4  Eq. 15 over the 3 x 3 rows of 3 cells around the
//                       particle (each row is one contiguous slot range; a
//                       lane per particle, two in small groups),
//                       amax per body by a labelled warp max + atomicMax
//   k_step          A5  limited step and tangential part; feature particles,
//                       and particles with no triangle within reach, finish
//                       here; the others are queued
//   k_search        A6  a group of lanes per queued particle over the
//                       triangles of the 27 cells: projection or revert;
//                       positions are written back in id order
#include <cfloat>

#include "body.h"

namespace fppg {

#ifdef FPPG_CHECKED
// the codes of the failed bounds checks since the last fppg_check_status
__device__ uint32_t g_check_word = 0u;
__device__ bool fppg_check_failed(uint32_t code) {
    atomicOr(&g_check_word, code);
    return false;
}
#endif

uint32_t check_word_take() {
#ifdef FPPG_CHECKED
    uint32_t w = 0u;
    const uint32_t zero = 0u;
    if (cudaMemcpyFromSymbol(&w, g_check_word, sizeof(w)) != cudaSuccess) return 0xffffffffu;
    cudaMemcpyToSymbol(g_check_word, &zero, sizeof(zero));
    return w;
#else
    return 0u;
#endif
}

namespace {

constexpr int TPB = 256;

inline unsigned nblocks(int64_t n, int t = TPB) { return (unsigned)std::max<int64_t>((n + t - 1) / t, 1); }

__device__ inline float3 f3(float4 a) { return make_float3(a.x, a.y, a.z); }
__device__ inline float3 operator-(float3 a, float3 b) { return make_float3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ inline float3 operator+(float3 a, float3 b) { return make_float3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ inline float3 operator*(float s, float3 a) { return make_float3(s * a.x, s * a.y, s * a.z); }
__device__ inline float dot3(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }

__device__ inline uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// max of v (>= 0) over the lanes that share `label`, added to dst[label] by
// one lane (dst starts every iteration at 0, so a max of 0 needs no atomic)
__device__ inline void labelled_max(uint32_t *dst, int label, float v) {
    uint32_t peers = __match_any_sync(0xffffffffu, label);
    uint32_t m = __reduce_max_sync(peers, __float_as_uint(v));
    if ((uint32_t)(__ffs(peers) - 1) == (threadIdx.x & 31u) && m) atomicMax(dst + label, m);
}

// The same over a whole block (every thread must call it): a warp whose
// lanes share one label leaves (label, max) in shared memory and thread 0
// adds one atomic per run of equal labels over the warps; a warp that
// mixes labels uses labelled_max.  On one large body this turns one
// same-address atomic per warp into one per block.
template <int WARPS>
__device__ inline void block_labelled_max(uint32_t *dst, int label, float v, int *s_lab, uint32_t *s_max) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int lab0 = __shfl_sync(0xffffffffu, label, 0);
    if (__all_sync(0xffffffffu, label == lab0)) {
        const uint32_t m = __reduce_max_sync(0xffffffffu, __float_as_uint(v));
        if (lane == 0) {
            s_lab[w] = lab0;
            s_max[w] = m;
        }
    } else {
        labelled_max(dst, label, v);
        if (lane == 0) {
            s_lab[w] = -1;
            s_max[w] = 0u;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int run_l = -1;
        uint32_t run_m = 0u;
        for (int q = 0; q < WARPS; q++) {
            if (s_lab[q] != run_l) {
                if (run_m) atomicMax(dst + run_l, run_m);
                run_l = s_lab[q];
                run_m = 0u;
            }
            if (run_l >= 0) run_m = max(run_m, s_max[q]);
        }
        if (run_m) atomicMax(dst + run_l, run_m);
    }
}

// the sort key: 8 (key_base + cell) + x-slab, with the grid row in the row order
__device__ inline uint32_t fine_key_of(const AsmParams &A, float x, float y, float z) {
    const int fx = fine_coord(x, A.ng_o[0], A.ng_inv, A.ng_n[0]);
    const int cy = cell_coord(y, A.ng_o[1], A.ng_inv, A.ng_n[1]);
    const int cz = cell_coord(z, A.ng_o[2], A.ng_inv, A.ng_n[2]);
    return kSlabs * A.key_base + (uint32_t)fx + kSlabs * (uint32_t)A.ng_n[0] * grid_row(A, cy, cz);
}

// ---- A1 ----------------------------------------------------------------------
__global__ void __launch_bounds__(TPB) k_keys(const float4 *__restrict__ pos, int64_t N,
                                              const AsmParams *__restrict__ P, uint32_t *__restrict__ key,
                                              uint32_t *__restrict__ amax, uint32_t *__restrict__ maxdisp, int B,
                                              uint32_t *__restrict__ work_count) {
    int64_t i = (int64_t)blockIdx.x * TPB + threadIdx.x;
    if (i < B) {
        amax[i] = 0u;
        maxdisp[i] = 0u;
    }
    if (i == 0) {
        work_count[0] = 0u;
        work_count[1] = 0u;
    }
    if (i >= N) return;
    float4 p = pos[i];
    key[i] = fine_key_of(P[body_of(p.w)], p.x, p.y, p.z);
}

// ---- A1-A3, counted form --------------------------------------------------------
// A counting sort over the dense fine keys: the keys are counted as they are
// made (every particle keeps its place in the arrival order of its key), the
// counts' exclusive scan is the start table itself, the ids go to start +
// arrival, and inside each key -- 2.2 particles on a lattice of spacing dx --
// the gather ranks them by id.  The result is the one order by (key, id),
// the same permutation as the stable sort of every key:
//   k_keys_count   keys, arrival places, counts per key
//   k_tile_sums    counts per tile of 4096 keys (more than kFewTiles tiles)
//   k_count_starts the start table from the counts; each block adds up what
//                  lies before it, so no block waits for another
//   k_place        ids by key, in arrival order; the counts back to 0
//   k_rank_gather  ids by (key, id); positions and constraints in that order
// A key shared by m particles costs each of them m comparisons, whatever their
// class: moving ones pay more for their pairs (and repel each other), but fixed
// ones have none.  So a set with fixed particles that puts more than kCrowd on
// one key is ordered by the radix form, which is linear; fixed particles stay
// where they are, so it is enough to look when the set is given or its classes
// are fixed (Group::find_crowds).  Iterations of 300,000 fixed particles, 512,
// 3,000 or all of them on a key: 74, 204 and 14,800 us, radix 86 each; of three
// million, 512 on a key: 407, radix 243; 20,000 loose ones: 36, radix 74.

__global__ void __launch_bounds__(TPB) k_keys_count(const float4 *__restrict__ pos, int64_t N,
                                                    const AsmParams *__restrict__ P, uint32_t *__restrict__ key,
                                                    uint32_t *__restrict__ place, uint32_t *__restrict__ cnt,
                                                    int64_t F) {
    const int64_t i = (int64_t)blockIdx.x * TPB + threadIdx.x;
    if (i >= N) return;
    const float4 p = pos[i];
    uint32_t k = fine_key_of(P[body_of(p.w)], p.x, p.y, p.z);
    if (!FPPG_CHECK(k < F, kChkGather)) k = 0u;
    key[i] = k;
    place[i] = atomicAdd(cnt + k, 1u);
}

// the counts of a tile of kCountTile keys as 16-byte vectors, vector q of a
// thread at keys f0 + 4 (q TPB + thread) .. + 3 (0 past F1)
constexpr int kCountVec = kCountTile / (4 * TPB);

__device__ inline uint4 load_counts(const uint32_t *__restrict__ cnt, int64_t f, int64_t F1) {
    if (f + 4 <= F1) return *reinterpret_cast<const uint4 *>(cnt + f);
    return make_uint4(f < F1 ? cnt[f] : 0u, f + 1 < F1 ? cnt[f + 1] : 0u, f + 2 < F1 ? cnt[f + 2] : 0u, 0u);
}

__device__ inline uint32_t sum4(const uint4 &a) { return a.x + a.y + a.z + a.w; }

__global__ void __launch_bounds__(TPB) k_tile_sums(const uint32_t *__restrict__ cnt, int64_t F1,
                                                   uint32_t *__restrict__ tiles) {
    __shared__ uint32_t wsum[TPB / 32];
    const int64_t f0 = (int64_t)blockIdx.x * kCountTile;
    uint32_t v = 0u;
#pragma unroll
    for (int q = 0; q < kCountVec; q++) v += sum4(load_counts(cnt, f0 + 4 * (q * TPB + (int)threadIdx.x), F1));
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int q = 1; q < TPB / 32; q++) v += wsum[q];
        tiles[blockIdx.x] = v;
    }
}

// fstart[f] = the number of particles with a fine key below f, for f in
// [0, F] (cnt: F1 = F + 1 entries, the last 0).  One tile per block, which
// adds up what lies before it: the tile sums (scanned = 0), one entry of
// their exclusive scan (scanned = 1), or with tiles null the counts
// themselves.  Also resets the per-body maxima and the search queue.
__global__ void __launch_bounds__(TPB) k_count_starts(const uint32_t *__restrict__ cnt,
                                                      const uint32_t *__restrict__ tiles, int scanned, int64_t F1,
                                                      uint32_t *__restrict__ fstart, uint32_t *__restrict__ amax,
                                                      uint32_t *__restrict__ maxdisp, int B,
                                                      uint32_t *__restrict__ work_count) {
    constexpr int kWarps = TPB / 32;
    static_assert(kCountVec * kWarps == 32, "one lane per (vector, warp) sum");
    __shared__ uint32_t s_sum[32], s_pre[kWarps];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t b = (int64_t)blockIdx.x * TPB + threadIdx.x; b < B; b += (int64_t)gridDim.x * TPB) {
        amax[b] = 0u;
        maxdisp[b] = 0u;
    }
    if (blockIdx.x == 0 && threadIdx.x < 2) work_count[threadIdx.x] = 0u;
    const int64_t f0 = (int64_t)blockIdx.x * kCountTile;
    uint4 v[kCountVec];
#pragma unroll
    for (int q = 0; q < kCountVec; q++) v[q] = load_counts(cnt, f0 + 4 * (q * TPB + (int)threadIdx.x), F1);
    uint32_t pre = 0u;   // this thread's share of what lies before the tile
    if (!tiles) {
        for (int64_t f = 4 * (int64_t)threadIdx.x; f < f0; f += 4 * TPB)
            pre += sum4(*reinterpret_cast<const uint4 *>(cnt + f));
    } else if (scanned) {
        if (threadIdx.x == 0) pre = tiles[blockIdx.x];
    } else {
#pragma unroll 4
        for (uint32_t t = threadIdx.x; t < blockIdx.x; t += TPB) pre += tiles[t];
    }
    pre = __reduce_add_sync(0xffffffffu, pre);
    if (lane == 0) s_pre[w] = pre;
    // inclusive sums over the warp of every vector
    uint32_t inc[kCountVec];
#pragma unroll
    for (int q = 0; q < kCountVec; q++) {
        inc[q] = sum4(v[q]);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc[q], o);
            if (lane >= o) inc[q] += t;
        }
        if (lane == 31) s_sum[q * kWarps + w] = inc[q];
    }
    __syncthreads();
    // every warp scans the 32 (vector, warp) sums for itself
    uint32_t all = s_sum[lane];
    const uint32_t own = all;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, all, o);
        if (lane >= o) all += t;
    }
    all -= own;
    uint32_t base = 0u;
#pragma unroll
    for (int q = 0; q < kWarps; q++) base += s_pre[q];
#pragma unroll
    for (int q = 0; q < kCountVec; q++) {
        const int64_t f = f0 + 4 * (q * TPB + (int)threadIdx.x);
        uint32_t r = base + __shfl_sync(0xffffffffu, all, q * kWarps + w) + inc[q] - sum4(v[q]);
        uint4 o;
        o.x = r;
        o.y = r += v[q].x;
        o.z = r += v[q].y;
        o.w = r += v[q].z;
        if (f + 4 <= F1) {
            *reinterpret_cast<uint4 *>(fstart + f) = o;
        } else {
            if (f < F1) fstart[f] = o.x;
            if (f + 1 < F1) fstart[f + 1] = o.y;
            if (f + 2 < F1) fstart[f + 2] = o.z;
        }
    }
}

// the counts alone, then their maximum where it passes kCrowd, and 0 again
__global__ void __launch_bounds__(TPB) k_crowd_counts(const float4 *__restrict__ pos, int64_t N,
                                                      const AsmParams *__restrict__ P, uint32_t *__restrict__ cnt,
                                                      int64_t F) {
    const int64_t i = (int64_t)blockIdx.x * TPB + threadIdx.x;
    if (i >= N) return;
    const float4 p = pos[i];
    const uint32_t k = fine_key_of(P[body_of(p.w)], p.x, p.y, p.z);
    if (FPPG_CHECK(k < F, kChkGather)) atomicAdd(cnt + k, 1u);
}

__global__ void __launch_bounds__(TPB) k_crowd_max(uint32_t *__restrict__ cnt, int64_t F1, uint32_t *__restrict__ most) {
    uint32_t m = 0u;
    const int64_t t = (int64_t)blockIdx.x * TPB + threadIdx.x, nv = F1 / 4;
    for (int64_t f = t; f < nv; f += (int64_t)gridDim.x * TPB) {
        const uint4 v = reinterpret_cast<const uint4 *>(cnt)[f];
        m = max(m, max(max(v.x, v.y), max(v.z, v.w)));
        reinterpret_cast<uint4 *>(cnt)[f] = make_uint4(0u, 0u, 0u, 0u);
    }
    if (t < F1 - 4 * nv) {
        m = max(m, cnt[4 * nv + t]);
        cnt[4 * nv + t] = 0u;
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0 && m > kCrowd) atomicMax(most, m);
}

// ids by key, in arrival order; the counts set back to 0 for the next build
__global__ void __launch_bounds__(TPB) k_place(const uint32_t *__restrict__ key, const uint32_t *__restrict__ place,
                                               const uint32_t *__restrict__ fstart, int64_t N,
                                               uint32_t *__restrict__ id_a, uint32_t *__restrict__ cnt, int64_t F1) {
    const int64_t i = (int64_t)blockIdx.x * TPB + threadIdx.x;
    const int64_t nv = F1 / 4;
    for (int64_t f = i; f < nv; f += (int64_t)gridDim.x * TPB)
        reinterpret_cast<uint4 *>(cnt)[f] = make_uint4(0u, 0u, 0u, 0u);
    if (i < F1 - 4 * nv) cnt[4 * nv + i] = 0u;
    if (i >= N || !FPPG_CHECK(key[i] < F1 - 1, kChkGather)) return;
    const uint32_t k = fstart[key[i]] + place[i];
    if (FPPG_CHECK(k < N, kChkGather)) id_a[k] = (uint32_t)i;
}

// One particle at slot k of the key order, written on its own: position,
// slot-pair halves, constraint, id
__device__ inline void put_slot(uint32_t k, const float4 &q, uint32_t id, int32_t c, int64_t N,
                                float4 *__restrict__ pos_s, float4 *__restrict__ pos_p, uint32_t *__restrict__ id_s,
                                int32_t *__restrict__ cons_s) {
    pos_s[k] = q;
    id_s[k] = id;
    cons_s[k] = c;
    float *a = reinterpret_cast<float *>(pos_p + (k >> 1)) + (k & 1u);
    float *b = reinterpret_cast<float *>(pos_p + (N + 1) / 2 + (k >> 1)) + (k & 1u);
    a[0] = q.x;
    a[2] = q.y;
    b[0] = q.z;
    b[2] = q.w;
}

// A block takes kGatherItems TPB consecutive places of the arrival order.
// Each particle is ranked by id among those of its key and goes to start +
// rank: within the block's slots through shared memory (stored coalesced),
// else -- a key that crosses the block's edge -- straight to its slot.  Bound
// by memory: 68 B per particle, with a chain of four dependent loads (id,
// position, start, the key's ids).  Two particles per thread keep more of
// them in flight once the blocks fill the chip (18.9 M particles: 278 -> 250
// us, 7.1 M: 107 -> 97 us); below that one (42 k: 3.1 against 3.9 us).  Grid build
// with one and two: 0.24 M 18.1 / 20.2 us, 0.51 M 24.3 / 24.9, 0.86 M 34.4 / 34.5,
// 1.16 M 43.1 / 42.9, 1.95 M 67.1 / 65.2, 4.0 M 124.8 / 120.5.
constexpr int64_t kGatherTwoMinN = 1 << 20;

template <int kGatherItems>
__global__ void __launch_bounds__(TPB) k_rank_gather(const uint32_t *__restrict__ id_a,
                                                     const AsmParams *__restrict__ P,
                                                     const uint32_t *__restrict__ fstart,
                                                     const float4 *__restrict__ pos, const int32_t *__restrict__ cons,
                                                     int64_t N, float4 *__restrict__ pos_s, float4 *__restrict__ pos_p,
                                                     uint32_t *__restrict__ id_s, int32_t *__restrict__ cons_s,
                                                     int64_t F) {
    constexpr int kGatherTile = kGatherItems * TPB;
    __shared__ float4 s_pos[kGatherTile];
    __shared__ uint32_t s_id[kGatherTile];
    __shared__ int32_t s_cons[kGatherTile];
    constexpr uint32_t kNone = 0xffffffffu;
    const int64_t k0 = (int64_t)blockIdx.x * kGatherTile;
    uint32_t id[kGatherItems], s[kGatherItems], e[kGatherItems];
    float4 q[kGatherItems];
    int32_t c[kGatherItems];
#pragma unroll
    for (int u = 0; u < kGatherItems; u++) {
        const int64_t k = k0 + u * TPB + threadIdx.x;
        s_id[u * TPB + threadIdx.x] = kNone;
        id[u] = k < N ? id_a[k] : kNone;
        if (k < N && !FPPG_CHECK(id[u] < N, kChkGather)) id[u] = kNone;
    }
#pragma unroll
    for (int u = 0; u < kGatherItems; u++)
        if (id[u] != kNone) {
            q[u] = pos[id[u]];
            c[u] = cons[id[u]];
        }
#pragma unroll
    for (int u = 0; u < kGatherItems; u++)
        if (id[u] != kNone) {
            // (the key again: cheaper than a gather of the stored one)
            const uint32_t f = fine_key_of(P[body_of(q[u].w)], q[u].x, q[u].y, q[u].z);
            if (FPPG_CHECK(f < F, kChkGather)) {
                s[u] = fstart[f];
                e[u] = fstart[f + 1u];
            } else {
                id[u] = kNone;
            }
        }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kGatherItems; u++) {
        if (id[u] == kNone) continue;
        uint32_t slot = s[u];
        if (e[u] - s[u] > 1u && FPPG_CHECK(s[u] <= e[u] && e[u] <= N, kChkGather))
            for (uint32_t j = s[u]; j < e[u]; j++) slot += id_a[j] < id[u] ? 1u : 0u;
        if (!FPPG_CHECK(slot < N, kChkGather)) continue;
        const int64_t l = (int64_t)slot - k0;
        if (l >= 0 && l < kGatherTile) {
            s_pos[l] = q[u];
            s_id[l] = id[u];
            s_cons[l] = c[u];
        } else {
            put_slot(slot, q[u], id[u], c[u], N, pos_s, pos_p, id_s, cons_s);
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kGatherItems; u++) {
        const int l = u * TPB + (int)threadIdx.x;
        const int64_t k = k0 + l;
        const uint32_t mine = s_id[l];
        // the padding of an odd count: a finite point of no class (its thread
        // is in the last block: an odd N is no multiple of the tile)
        const bool pad = k == N && (N & 1);
        const bool here = mine != kNone || pad;
        const float4 v = mine != kNone ? s_pos[l] : make_float4(0.f, 0.f, 0.f, 0.f);
        if (mine != kNone) {
            pos_s[k] = v;
            id_s[k] = mine;
            cons_s[k] = s_cons[l];
        }
        // slot pairs: the two slots sit in neighbouring lanes, which swap
        // their points and write one half each (as in k_gather); a slot whose
        // partner is written elsewhere writes its own four values
        const float ox = __shfl_xor_sync(0xffffffffu, v.x, 1), oy = __shfl_xor_sync(0xffffffffu, v.y, 1);
        const float oz = __shfl_xor_sync(0xffffffffu, v.z, 1), ow = __shfl_xor_sync(0xffffffffu, v.w, 1);
        const bool both = __shfl_xor_sync(0xffffffffu, here ? 1 : 0, 1) != 0 && here;
        if (both) {
            if ((k & 1) == 0) pos_p[k >> 1] = make_float4(v.x, ox, v.y, oy);
            else pos_p[(N + 1) / 2 + (k >> 1)] = make_float4(oz, v.z, ow, v.w);
        } else if (here) {
            float *a = reinterpret_cast<float *>(pos_p + (k >> 1)) + (k & 1);
            float *b = reinterpret_cast<float *>(pos_p + (N + 1) / 2 + (k >> 1)) + (k & 1);
            a[0] = v.x;
            a[2] = v.y;
            b[0] = v.z;
            b[2] = v.w;
        }
    }
}

// the sorted keys (diagnostics)
__global__ void __launch_bounds__(TPB) k_sorted_keys(const uint32_t *__restrict__ id_s,
                                                     const uint32_t *__restrict__ key, int64_t N,
                                                     uint32_t *__restrict__ out) {
    const int64_t k = (int64_t)blockIdx.x * TPB + threadIdx.x;
    if (k < N) out[k] = key[id_s[k]];
}

// ---- A3 ----------------------------------------------------------------------
// Positions in key order (also as slot pairs) and the constraint ids in key
// order.
__global__ void __launch_bounds__(TPB) k_gather(const uint32_t *__restrict__ id_s, const float4 *__restrict__ pos,
                                                int64_t N, float4 *__restrict__ pos_s, float4 *__restrict__ pos_p,
                                                const int32_t *__restrict__ cons, int32_t *__restrict__ cons_s) {
    const int64_t k = (int64_t)blockIdx.x * TPB + threadIdx.x;
    const bool valid = k < N;
    uint32_t id = valid ? id_s[k] : 0u;
    if (valid && !FPPG_CHECK(id < N, kChkGather)) id = 0u;
    const float4 q = valid ? pos[id] : make_float4(0.f, 0.f, 0.f, 0.f);
    // the constraint ids in key order too, for the step
    if (valid && cons_s) cons_s[k] = cons[id];
    // slot-pair copy: pair m = slots 2m and 2m + 1 as {x0, x1, y0, y1} at
    // pos_p[m] and {z0, z1, w0, w1} at pos_p[(N + 1) / 2 + m]; the two slots
    // sit in neighbouring lanes, which swap their points and write one half
    // each; past the last slot a lane holds a finite point of no class, the
    // padding of an odd count
    const float ox = __shfl_xor_sync(0xffffffffu, q.x, 1), oy = __shfl_xor_sync(0xffffffffu, q.y, 1);
    const float oz = __shfl_xor_sync(0xffffffffu, q.z, 1), ow = __shfl_xor_sync(0xffffffffu, q.w, 1);
    if ((k & 1) == 0) {
        if (valid) pos_p[k >> 1] = make_float4(q.x, ox, q.y, oy);
    } else if (k <= N) {
        pos_p[(N + 1) / 2 + (k >> 1)] = make_float4(oz, q.z, ow, q.w);
    }
    if (valid) pos_s[k] = q;
}

// The dense start table of the fine keys, from the sorted keys themselves:
// fstart[f] = the first slot whose fine key is >= f, for f in [0, F] (so
// fstart[F] = N).  The fine keys are cut into blocks of kStartBlock.
// k_key_block_starts: slot k starts the blocks (b(k - 1), b(k)] (b = key /
// kStartBlock; block -1 before the first slot, the block count after the
// last), so each block's first slot is written once, by the slot whose key
// step crosses it.  k_fine_starts: one CTA per block; the block's slots
// [bstart[b], bstart[b + 1]) hold every key of the block, and each thread
// finds its fine key's lower bound among them by binary search, in shared
// memory when the slots fit.  Every entry is written once: no counts,
// atomics or scans.  (Tiles of 4096 fine keys with a 16-key walk per
// thread measured slower: the table of the largest workload, 63 MB, stays
// in L2 either way, and the short per-thread search keeps more loads in
// flight.)
constexpr int kStartStage = 4096;

__global__ void __launch_bounds__(TPB) k_key_block_starts(const uint32_t *__restrict__ key_s, int64_t N,
                                                          int64_t nblk, uint32_t *__restrict__ bstart) {
    const int64_t k = (int64_t)blockIdx.x * TPB + threadIdx.x;
    if (k > N) return;
    int64_t b0 = k == 0 ? -1 : (int64_t)(key_s[k - 1] / kStartBlock);
    int64_t b1 = k == N ? nblk : (int64_t)(key_s[k] / kStartBlock);
    if (!FPPG_CHECK(b0 < nblk && b1 <= nblk, kChkGather)) {   // a key past the fine-key count
        b0 = min(b0, nblk - 1);
        b1 = min(b1, nblk);
    }
    for (int64_t b = b0 + 1; b <= b1; b++) bstart[b] = (uint32_t)k;
}

__global__ void __launch_bounds__(kStartBlock) k_fine_starts(const uint32_t *__restrict__ key_s,
                                                             const uint32_t *__restrict__ bstart, int64_t F1,
                                                             uint32_t *__restrict__ fstart) {
    __shared__ uint32_t s_key[kStartStage];
    const int64_t b = blockIdx.x;
    const uint32_t lo = bstart[b], hi = bstart[b + 1];
    const uint32_t len = hi > lo ? hi - lo : 0u;
    const bool staged = len <= (uint32_t)kStartStage;
    if (staged)
        for (uint32_t i = threadIdx.x; i < len; i += kStartBlock) s_key[i] = key_s[lo + i];
    __syncthreads();
    const int64_t f = b * kStartBlock + threadIdx.x;
    if (f >= F1) return;
    uint32_t a = 0u, c = len;   // first of the block's slots with key >= f
    while (a < c) {
        const uint32_t m = (a + c) >> 1;
        if ((int64_t)(staged ? s_key[m] : key_s[lo + m]) < f) a = m + 1u;
        else c = m;
    }
    fstart[f] = lo + a;
}

// ---- A4 ----------------------------------------------------------------------
// a_i = -sum_j dW/dr(r_ij) e_ij = force_scale * sum_j (1 - r_ij / 2h)^3 (x_i - x_j)
//
// Each lane owns one particle (key order) and scans the 3 x 3 grid rows
// around it; per row it walks one contiguous slot range: the x-slabs of the
// row's stencil cells that lie within the reach sqrt((2h)^2 - gap_y^2 -
// gap_z^2) of it (rows out of reach are skipped).  Candidates come two at a
// time from the slot-pair copy pos_p ({x0, x1, y0, y1}, {z0, z1, w0, w1}),
// so one float4 load gives the packed FP32x2 operands; each packed
// operation is per component identical to the scalar round-to-nearest one,
// so the neighbour test r^2 = (dx dx + dy dy) + dz dz < (2h)^2 decides
// exactly as the scalar rule.  The loop works on q - p (the exact negation
// of p - q) and accumulates without branches into two partial sums.
//
// Variant 0 walks each lane's own ranges.  Variant 1 (shared row): when
// every moving lane of a warp lies in the same grid row of the same body,
// the lanes' ranges for one row offset lie in a single grid row and the
// warp walks their union in lockstep (broadcast loads); a candidate outside
// a lane's own range is out of its reach and fails the test.
// The particle itself adds (1 - 0)^3 * 0 = 0, so no self test is needed.
// Slots are paired by absolute parity (even -> .x, odd -> .y) with the range
// [s, e) applied as a mask, so every accepted neighbour lands in the same
// partial sum, in the same order, in every variant.
// COUNT adds, per particle, the accepted neighbours (self excluded) and the
// slots of its own ranges (candidates tested).
// r = sqrt(r^2) by sqrt_approx (exactly 0 at 0, so the particle itself
// needs no guard)

struct PairAcc {
    float2 ax, ay, az;
    int cnt;
};

// One slot pair (2m, 2m + 1).  EDGE: the pair may hold a slot outside the
// range [s, e) (the first and last pair of a range), which is masked out.
// The weight is clamped at zero, max(1 - r / 2h, 0)^3, instead of testing
// r^2 < (2h)^2: a pair beyond 2h adds exactly 0, one within rounding of 2h a
// weight below 1e-18; unless every class acts on the lane (ALL) the class
// mask selects.  The counting form keeps the exact FP32 test.
// pos_p holds the {x, y} halves of the slot pairs, pos_b the {z, w} halves;
// where every class acts on the lane (ALL) the class bits are not needed and
// only {z0, z1} is read: 24 bytes per slot pair instead of 32.
template <bool ALL, bool COUNT, bool EDGE>
__device__ inline void pair_step(const float4 *__restrict__ pos_p, const float4 *__restrict__ pos_b, uint32_t m,
                                 uint32_t s, uint32_t e, const float2 npx, const float2 npy, const float2 npz,
                                 uint32_t mbits, float R2, float hih, PairAcc &acc, uint32_t self) {
    const uint32_t j = 2 * m;
    const bool has0 = !EDGE || j >= s, has1 = !EDGE || j + 1 < e;
    const float4 A = pos_p[m];
    float4 B;
    if (ALL) {
        const float2 z = *reinterpret_cast<const float2 *>(pos_b + m);
        B = make_float4(z.x, z.y, 0.f, 0.f);
    } else {
        B = pos_b[m];
    }
    const float2 dx = __fadd2_rn(make_float2(A.x, A.y), npx);     // q - p
    const float2 dy = __fadd2_rn(make_float2(A.z, A.w), npy);
    const float2 dz = __fadd2_rn(make_float2(B.x, B.y), npz);
    float2 w;
    if (!COUNT) {
        // r^2 with fused multiply-adds and the weight max(1 - r / 2h, 0)^3
        // from a saturating FMA: no decision is taken on r^2 here (a slot
        // beyond 2h weighs exactly 0, one within rounding of 2h below 1e-18)
        const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
        const float2 t = make_float2(__saturatef(fmaf(sqrt_approx(r2.x), -hih, 1.f)),
                                     __saturatef(fmaf(sqrt_approx(r2.y), -hih, 1.f)));
        w = __fmul2_rn(__fmul2_rn(t, t), t);
        bool k0 = has0, k1 = has1;
        if (!ALL) {
            k0 = k0 && (mbits & __float_as_uint(B.z)) != 0u;
            k1 = k1 && (mbits & __float_as_uint(B.w)) != 0u;
        }
        if (EDGE || !ALL) {
            w.x = k0 ? w.x : 0.f;
            w.y = k1 ? w.y : 0.f;
        }
    } else {
        // the counting form: the exact FP32 test r^2 = (dx dx + dy dy) + dz dz
        // < (2h)^2 without contraction decides each neighbour
        const float2 r2 = __fadd2_rn(__fadd2_rn(__fmul2_rn(dx, dx), __fmul2_rn(dy, dy)), __fmul2_rn(dz, dz));
        const float2 r = make_float2(sqrt_approx(r2.x), sqrt_approx(r2.y));
        const float2 t = __ffma2_rn(r, make_float2(-hih, -hih), make_float2(1.f, 1.f));   // 1 - r / 2h
        bool t0 = has0 && r2.x < R2, t1 = has1 && r2.y < R2;
        if (!ALL) {
            t0 = t0 && (mbits & __float_as_uint(B.z)) != 0u;
            t1 = t1 && (mbits & __float_as_uint(B.w)) != 0u;
        }
        if (COUNT) acc.cnt += (int)(t0 && j != self) + (int)(t1 && j + 1 != self);
        w = __fmul2_rn(__fmul2_rn(t, t), t);
        w.x = t0 ? w.x : 0.f;
        w.y = t1 ? w.y : 0.f;
    }
    acc.ax = __ffma2_rn(w, dx, acc.ax);
    acc.ay = __ffma2_rn(w, dy, acc.ay);
    acc.az = __ffma2_rn(w, dz, acc.az);
}

// the slot pairs [s >> 1, (e + 1) >> 1) of range [s, e): the first and last
// pair masked, the ones between without a range test
template <bool ALL, bool COUNT>
__device__ inline void force_range2(const float4 *__restrict__ pos_p, const float4 *__restrict__ pos_b,
                                    const float2 npx, const float2 npy, const float2 npz, uint32_t mbits, float R2,
                                    float hih, uint32_t s, uint32_t e, PairAcc &acc, uint32_t self) {
    if (s >= e) return;
    uint32_t m = s >> 1;
    const uint32_t m1 = (e + 1) >> 1;
    pair_step<ALL, COUNT, true>(pos_p, pos_b, m, s, e, npx, npy, npz, mbits, R2, hih, acc, self);
    if (m + 1 >= m1) return;
    for (m = m + 1; m + 1 < m1; m++)
        pair_step<ALL, COUNT, false>(pos_p, pos_b, m, s, e, npx, npy, npz, mbits, R2, hih, acc, self);
    pair_step<ALL, COUNT, true>(pos_p, pos_b, m1 - 1, s, e, npx, npy, npz, mbits, R2, hih, acc, self);
}

// k_force with two lanes a particle.  Particles up to which it is taken: a
// lane's walk of ~350 slots is the launch's length while the warps do not fill
// the chip.  One lane -> two: 42 k particles 35.9 -> 19.8 us, 76 k 31.5 -> 27.3,
// 540 k 121 -> 155, 777 k 166 -> 216; the lines through the last three cross
// at about 125 k.
constexpr int64_t kSplitMaxN = 100000;

// every second slot of [j, e): the operations of pair_step (not COUNT) on one
// half, in the same order
__device__ inline void force_slots(const float4 *__restrict__ pos_s, const float4 &p, uint32_t mbits, float hih,
                                   uint32_t j, uint32_t e, float sum[3]) {
#pragma unroll 4
    for (; j < e; j += 2) {
        const float4 q = pos_s[j];
        const float dx = __fadd_rn(q.x, -p.x), dy = __fadd_rn(q.y, -p.y), dz = __fadd_rn(q.z, -p.z);
        const float r2 = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
        const float t = __saturatef(__fmaf_rn(sqrt_approx(r2), -hih, 1.f));
        const float w = (mbits & __float_as_uint(q.w)) != 0u ? __fmul_rn(__fmul_rn(t, t), t) : 0.f;
        sum[0] = __fmaf_rn(w, dx, sum[0]);
        sum[1] = __fmaf_rn(w, dy, sum[1]);
        sum[2] = __fmaf_rn(w, dz, sum[2]);
    }
}

// SPLIT (variant 0 without counts): two lanes a particle, one for the even and
// one for the odd slots.  The one-lane form sums these apart, in the halves of
// its packed sums, and adds the two at the end; so both forms give the same
// bits.  A lane's step takes one candidate instead of two: a walk 1.8 times
// shorter for 1.3 times the work.
template <int VARIANT, bool COUNT, bool MORTON, bool SPLIT>
// (at most 48 registers: five 256-thread blocks per SM; 80 in the split form,
// whose groups do not fill the chip)
__global__ void __launch_bounds__(TPB, SPLIT ? 3 : 5)
    k_force(const float4 *__restrict__ pos_s, const float4 *__restrict__ pos_p, int64_t N,
            const AsmParams *__restrict__ P, const uint32_t *__restrict__ fstart, float4 *__restrict__ acc_s,
            uint32_t *__restrict__ amax, int32_t *__restrict__ count_s, int32_t *__restrict__ tested_s) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, k = SPLIT ? t >> 1 : t;
    const uint32_t half = threadIdx.x & 1u;
    const bool active = k < N;
    const float4 p = active ? pos_s[k] : make_float4(0.f, 0.f, 0.f, 0.f);
    const int cls = active ? cls_of(p.w) : kClsI;
    const int b = active ? body_of(p.w) : 0;
    const AsmParams &A = P[b];
    const bool mob = active && is_mobile(cls, A) && !is_ghost(p.w);
    // the counting form also counts the neighbours of fixed particles
    const uint32_t mbits = (mob || (COUNT && active)) ? acts_on_bits(cls) : 0u;
    const int nx = A.ng_n[0], ny = A.ng_n[1], nz = A.ng_n[2];
    const GridPoint g = grid_point(A, p.x, p.y, p.z);
    const int cy = g.c[1], cz = g.c[2];
    const float R2 = A.R2, hih = A.half_inv_h;
    const float2 npx = make_float2(-p.x, -p.x), npy = make_float2(-p.y, -p.y), npz = make_float2(-p.z, -p.z);
    const float4 *pos_b = pos_p + (N + 1) / 2;
    // every class acts on every moving lane (volume targets): no mask test
    const bool all_cls = __all_sync(0xffffffffu, mbits == 0u || mbits == 0x1Fu);
    bool shared_row = false;
    if (VARIANT == 1) {
        const uint32_t mover = __ballot_sync(0xffffffffu, mbits != 0u);
        const int leader = mover ? __ffs(mover) - 1 : 0;
        const uint32_t rowkey = A.key_base + (uint32_t)nx * grid_row_of<MORTON>(A, cy, cz);
        const uint32_t lead_row = __shfl_sync(0xffffffffu, rowkey, leader);
        shared_row = __all_sync(0xffffffffu, mbits == 0u || rowkey == lead_row);
    }
    float sum[3] = {0.f, 0.f, 0.f};
    PairAcc acc{make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), 0};
    int tested = 0;
    for (int dz = -1; dz <= 1; dz++) {
        const int z = cz + dz;
        const float gz = row_gap(g.t[2], cz, dz, g.slack);
        for (int dy = -1; dy <= 1; dy++) {
            const int y = cy + dy;
            uint32_t s = 0xffffffffu, e = 0u;
            if (mbits && z >= 0 && z < nz && y >= 0 && y < ny) {
                const uint32_t row = A.key_base + (uint32_t)nx * grid_row_of<MORTON>(A, y, z);
                row_slots(A, fstart, g, row_gap(g.t[1], cy, dy, g.slack), gz, row, s, e);
                if (!FPPG_CHECK(e == 0u || (s <= e && e <= (uint64_t)N), kChkRange)) {
                    s = 0xffffffffu;
                    e = 0u;
                }
            }
            if (COUNT && e > s) tested += (int)(e - s);
            if (VARIANT == 1 && shared_row) {
                s = __reduce_min_sync(0xffffffffu, s);
                e = __reduce_max_sync(0xffffffffu, e);
            }
            if (SPLIT)
                force_slots(pos_s, p, mbits, hih, s + ((s ^ half) & 1u), e, sum);
            else if (all_cls)
                force_range2<true, COUNT>(pos_p, pos_b, npx, npy, npz, mbits, R2, hih, s, e, acc, (uint32_t)k);
            else
                force_range2<false, COUNT>(pos_p, pos_b, npx, npy, npz, mbits, R2, hih, s, e, acc, (uint32_t)k);
        }
    }
    if (SPLIT) {
        acc.ax = make_float2(sum[0], __shfl_xor_sync(0xffffffffu, sum[0], 1));
        acc.ay = make_float2(sum[1], __shfl_xor_sync(0xffffffffu, sum[1], 1));
        acc.az = make_float2(sum[2], __shfl_xor_sync(0xffffffffu, sum[2], 1));
    }
    float fx = 0.f, fy = 0.f, fz = 0.f, mag = 0.f;
    if (mob) {
        // the sums hold q - p: negate
        fx = -(acc.ax.x + acc.ax.y) * A.force_scale;
        fy = -(acc.ay.x + acc.ay.y) * A.force_scale;
        fz = -(acc.az.x + acc.az.y) * A.force_scale;
        mag = sqrtf(fx * fx + fy * fy + fz * fz);
    }
    if (active && (!SPLIT || half == 0u)) acc_s[k] = make_float4(fx, fy, fz, mag);
    if (COUNT && active) {
        count_s[k] = acc.cnt;
        if (tested_s) tested_s[k] = mob ? tested : 0;
    }
    labelled_max(amax, A.amax_slot, mag);
}

// Masked neighbour count (self excluded) and the number of candidates in the
// particle's own 27 cells (the full stencil, no reach cut), per particle in
// key order (diagnostics).
__global__ void __launch_bounds__(TPB) k_count(const float4 *__restrict__ pos_s, int64_t N,
                                               const AsmParams *__restrict__ P, const uint32_t *__restrict__ fstart,
                                               int32_t *__restrict__ count_s, int32_t *__restrict__ cand_s) {
    const int64_t k = (int64_t)blockIdx.x * TPB + threadIdx.x;
    if (k >= N) return;
    const float4 p = pos_s[k];
    const int cls = cls_of(p.w);
    const AsmParams &A = P[body_of(p.w)];
    const uint32_t mbits = acts_on_bits(cls);
    const int nx = A.ng_n[0], ny = A.ng_n[1], nz = A.ng_n[2];
    const int cx = cell_coord(p.x, A.ng_o[0], A.ng_inv, nx);
    const int cy = cell_coord(p.y, A.ng_o[1], A.ng_inv, ny);
    const int cz = cell_coord(p.z, A.ng_o[2], A.ng_inv, nz);
    int cnt = 0, cand = 0;
    for (int z = max(cz - 1, 0); z <= min(cz + 1, nz - 1); z++)
        for (int y = max(cy - 1, 0); y <= min(cy + 1, ny - 1); y++) {
            const uint32_t row = A.key_base + (uint32_t)nx * grid_row(A, y, z);
            uint32_t s, e;
            cells_slots(fstart, row, max(cx - 1, 0), min(cx + 1, nx - 1), s, e);
            if (e > s) cand += (int)(e - s);
            for (uint32_t j = s; j < e; j++) {
                const float4 q = pos_s[j];
                const float r2 = dist2_rn(p.x - q.x, p.y - q.y, p.z - q.z);
                if (r2 < A.R2 && (int64_t)j != k && (mbits & __float_as_uint(q.w)) != 0u) cnt++;
            }
        }
    if (count_s) count_s[k] = cnt;
    if (cand_s) cand_s[k] = is_mobile(cls, A) && !is_ghost(p.w) ? cand : 0;
}

// ---- A6 helpers -------------------------------------------------------------

// closest point on a triangle by barycentric regions (Ericson, Real-Time
// Collision Detection, 2005); region 0 face, 1 + k edge (v_k, v_k+1),
// 4 + k vertex k
__device__ inline float3 closest_on_triangle(float3 p, float3 a, float3 b, float3 c, int &region) {
    const float3 ab = b - a, ac = c - a, ap = p - a;
    const float d1 = dot3(ab, ap), d2 = dot3(ac, ap);
    if (d1 <= 0.f && d2 <= 0.f) {
        region = 4;
        return a;
    }
    const float3 bp = p - b;
    const float d3 = dot3(ab, bp), d4 = dot3(ac, bp);
    if (d3 >= 0.f && d4 <= d3) {
        region = 5;
        return b;
    }
    const float vc = d1 * d4 - d3 * d2;
    if (vc <= 0.f && d1 >= 0.f && d3 <= 0.f) {
        region = 1;
        return a + (d1 / (d1 - d3)) * ab;
    }
    const float3 cp = p - c;
    const float d5 = dot3(ab, cp), d6 = dot3(ac, cp);
    if (d6 >= 0.f && d5 <= d6) {
        region = 6;
        return c;
    }
    const float vb = d5 * d2 - d1 * d6;
    if (vb <= 0.f && d2 >= 0.f && d6 <= 0.f) {
        region = 3;
        return a + (d2 / (d2 - d6)) * ac;
    }
    const float va = d3 * d6 - d5 * d4;
    if (va <= 0.f && (d4 - d3) >= 0.f && (d5 - d6) >= 0.f) {
        region = 2;
        return b + ((d4 - d3) / ((d4 - d3) + (d5 - d6))) * (c - b);
    }
    const float den = 1.f / (va + vb + vc);
    region = 0;
    return a + (vb * den) * ab + (vc * den) * ac;
}

// Search of the 27 triangle cells around y by a group of G neighbouring lanes
// (1, 8 or 32; every lane of the group holds the same y): each lane tests
// every G-th candidate, and the group reduces to the overall best with ties to
// the lower triangle index, so the choice is the same as a serial scan of the
// 27 cells, for every G.
//   surface: smallest |plane distance| among triangles whose foot is inside
//            (edge functions >= 0); returns the triangle or -1
//   volume:  closest triangle; returns inside (sign of (y - c) . psi <= 0)
//            or true when no triangle is near
struct CellRange {
    uint32_t beg, len;
};

// cell c < 27 of the block around y
__device__ inline CellRange block_cell(const MeshView &M, const AsmParams &A, float3 y, int c) {
    CellRange r{0u, 0u};
    const int x = cell_coord(y.x, A.tg_o[0], A.tg_inv, A.tg_n[0]) + c % 3 - 1;
    const int yy = cell_coord(y.y, A.tg_o[1], A.tg_inv, A.tg_n[1]) + (c / 3) % 3 - 1;
    const int z = cell_coord(y.z, A.tg_o[2], A.tg_inv, A.tg_n[2]) + c / 9 - 1;
    if (x < 0 || yy < 0 || z < 0 || x >= A.tg_n[0] || yy >= A.tg_n[1] || z >= A.tg_n[2]) return r;
    if (!test_bit(M.occ, A.occ_off, tri_key(A, x, yy, z))) return r;
    tri_cell(M, A, x, yy, z, r.beg, r.len);
    return r;
}

// the lanes of this lane's group, and its place in it
template <int G>
__device__ inline uint32_t group_mask() {
    return G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << (threadIdx.x & 31u & ~(uint32_t)(G - 1));
}
template <int G>
__device__ inline int group_lane() {
    return (int)(threadIdx.x & (uint32_t)(G - 1));
}

// lexicographic (value, index) minimum over the group; every lane gets it
template <int G>
__device__ inline void group_argmin(float &v, int &t) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(group_mask<G>(), v, o);
        const int ot = __shfl_xor_sync(group_mask<G>(), t, o);
        if (ov < v || (ov == v && ot < t)) {
            v = ov;
            t = ot;
        }
    }
}

// Surface candidate test: the foot of y on the plane of triangle t lies
// inside it (every in-plane edge distance >= -edge_tol: Fig. 8 with a
// tolerance, so a foot on a shared edge belongs to both triangles); *d gets
// the signed plane distance
__device__ inline bool surface_candidate(const MeshView &M, const AsmParams &A, int t, float3 y, float &d) {
    const float4 *g = M.geo + 5 * (size_t)(A.tri_off + t);
    const float3 u = y - f3(g[0]);
    const float tol = -A.edge_tol;
    const float4 m0 = g[2];
    if (dot3(u, f3(m0)) < tol) return false;
    const float4 m1 = g[3];
    if (dot3(u, f3(m1)) - m1.w < tol) return false;
    const float4 m2 = g[4];
    if (dot3(u, f3(m2)) - m2.w < tol) return false;
    d = dot3(u, f3(g[1]));
    return true;
}

// The same decision, with every edge evaluated: *emin gets the smallest
// in-plane edge distance of the foot (negative outside), so a triangle that
// is not projectable at y stays so within -emin - edge_tol of y (the edge
// distances are 1-Lipschitz in y: unit in-plane edge normals)
__device__ inline bool surface_candidate_margin(const MeshView &M, const AsmParams &A, int t, float3 y, float &d,
                                                float &emin) {
    const float4 *g = M.geo + 5 * (size_t)(A.tri_off + t);
    const float3 u = y - f3(g[0]);
    const float tol = -A.edge_tol;
    const float4 m0 = g[2], m1 = g[3], m2 = g[4];
    const float e0 = dot3(u, f3(m0));
    const float e1 = dot3(u, f3(m1)) - m1.w;
    const float e2 = dot3(u, f3(m2)) - m2.w;
    emin = fminf(e0, fminf(e1, e2));
    if (e0 < tol || e1 < tol || e2 < tol) return false;
    d = dot3(u, f3(g[1]));
    return true;
}

// Surface certificate (not in the paper; it changes no decision): when
// exactly one candidate is projectable at y, every other candidate of y's
// triangle cell stays non-projectable within the smallest -emin - edge_tol
// over them, so for a trial point in the same cell and within that radius
// the choice is the particle's own triangle if it is projectable there, and
// the step takes it without the search.  Radius shrunk by 2^-10 relative and
// 2^-12 dx for the FP32 rounding of the edge distances; 0: no certificate.
__device__ inline float surface_cert_radius(const AsmParams &A, int n_projectable, float r_other) {
    if (n_projectable != 1 || !(r_other < FLT_MAX)) return 0.f;
    return fmaxf(r_other * (1.f - 0x1p-10f) - A.dx * 0x1p-12f, 0.f);
}

// The candidate triangles of the 27 cells around triangle cell c as a range
// [beg, end) of M.cand (built with the mesh: the distinct triangles of the 27
// cells), (0, 0) for no triangle, (kProbeCells, kProbeCells) for a list too long
// to build.  The step computes it for every particle it queues, so that the
// search starts from the list instead of the chain bitmap -> rank -> list start.
constexpr uint32_t kProbeCells = 0xffffffffu;

__device__ inline uint2 cand_range(const MeshView &M, const AsmParams &A, uint32_t c) {
    const uint32_t w = M.occ[A.dil_off + (c >> 5)];
    if (!((w >> (c & 31u)) & 1u)) return make_uint2(0u, 0u);
    const uint32_t r = M.drank[A.drank_off + (c >> 5)] + __popc(w & ((1u << (c & 31u)) - 1u));
    const uint32_t o0 = M.coff[A.coff_off + r], o1 = M.coff[A.coff_off + r + 1];
    if (o0 >> 31) return make_uint2(kProbeCells, kProbeCells);
    return make_uint2(A.cand_off + o0, A.cand_off + (o1 & 0x7fffffffu));
}

__device__ inline uint32_t tri_cell_of(const AsmParams &A, float3 y) {
    return tri_key(A, cell_coord(y.x, A.tg_o[0], A.tg_inv, A.tg_n[0]), cell_coord(y.y, A.tg_o[1], A.tg_inv, A.tg_n[1]),
                   cell_coord(y.z, A.tg_o[2], A.tg_inv, A.tg_n[2]));
}

// the candidates of y's cell: 1 with [beg, end) into M.cand, 2 for cells to be
// probed, 0 for none; the same for every lane of a group, which holds one y.
// pre: the range of y's cell when the caller has it (nullptr: look it up)
__device__ inline int cell_candidates(const MeshView &M, const AsmParams &A, float3 y, uint32_t &beg, uint32_t &end,
                                      const uint2 *pre = nullptr) {
    const uint2 r = pre ? *pre : cand_range(M, A, tri_cell_of(A, y));
    if (r.x == kProbeCells) return 2;
    if (r.y <= r.x) return 0;
    beg = r.x;
    end = r.y;
    return 1;
}

// every candidate triangle of the 27 cells around y (of y's own cell alone
// with own_cell), spread over the group's lanes
template <int G, typename Test>
__device__ inline void for_27_candidates(const MeshView &M, const AsmParams &A, float3 y, bool own_cell, Test &&test,
                                         const uint2 *pre = nullptr) {
    const int sub = group_lane<G>();
    uint32_t beg = 0, end = 0;
    const int kind = own_cell ? 3 : cell_candidates(M, A, y, beg, end, pre);
    auto checked = [&](int t) {
        if (FPPG_CHECK(t >= 0 && t < A.nt, kChkTri)) test(t);
    };
    if (kind == 1) {
        for (uint32_t q = beg + sub; q < end; q += G) checked(M.cand[q]);
    } else if (kind == 2) {
        // (these cells hold over 512 entries together: the lanes look the
        // cells up side by side, then share out every cell's list)
        for (int c0 = 0; c0 < 27; c0 += G) {
            const CellRange r = c0 + sub < 27 ? block_cell(M, A, y, c0 + sub) : CellRange{0u, 0u};
            for (int k = 0; k < G && c0 + k < 27; k++) {
                const uint32_t b = G > 1 ? __shfl_sync(group_mask<G>(), r.beg, k, G) : r.beg;
                const uint32_t l = G > 1 ? __shfl_sync(group_mask<G>(), r.len, k, G) : r.len;
                for (uint32_t e = b + sub; e < b + l; e += G) checked(M.tlist[e]);
            }
        }
    } else if (kind == 3) {
        const CellRange r = block_cell(M, A, y, 13);
        for (uint32_t e = r.beg + sub; e < r.beg + r.len; e += G) checked(M.tlist[e]);
    }
}

// closest projectable triangle (smallest |plane distance|, ties to the lower
// index) among those binned into the 27 cells around y, or into y's own
// cell alone (own_cell); -1 when none
template <int G>
__device__ int group_project_surface(const MeshView &M, const AsmParams &A, float3 y, float &dist,
                                     bool own_cell = false, const uint2 *pre = nullptr, float *cert_r = nullptr) {
    float best = FLT_MAX, bd = 0.f;
    int bt = 0x7fffffff;
    int nproj = 0;
    float rother = FLT_MAX;
    for_27_candidates<G>(M, A, y, own_cell, [&](int t) {
        float d;
        if (cert_r) {
            float emin;
            if (!surface_candidate_margin(M, A, t, y, d, emin)) {
                rother = fminf(rother, -emin - A.edge_tol);
                return;
            }
            nproj++;
        } else if (!surface_candidate(M, A, t, y, d)) {
            return;
        }
        const float ad = fabsf(d);
        if (ad < best || (ad == best && t < bt)) {
            best = ad;
            bt = t;
            bd = d;
        }
    }, pre);
    float v = best;
    int t = bt;
    group_argmin<G>(v, t);
    dist = bd;
    if (G > 1) {
        // the signed distance of the winner, from a lane that holds it
        const uint32_t own = __ballot_sync(group_mask<G>(), bt == t && best == v) & group_mask<G>();
        dist = __shfl_sync(group_mask<G>(), bd, own ? __ffs(own) - 1 : 0);
    }
    if (cert_r) {
        float r = rother;
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
            r = fminf(r, __shfl_xor_sync(group_mask<G>(), r, o));
            nproj += __shfl_xor_sync(group_mask<G>(), nproj, o);
        }
        *cert_r = surface_cert_radius(A, nproj, r);
    }
    return t == 0x7fffffff ? -1 : t;
}

// Surface re-projection of trial point y of a particle on triangle c: the
// closest projectable triangle over the 27 cells, or with A.cascade the
// cascade of Sec. 3.3.3 (still on triangle c: stay; else the closest
// projectable one of y's own cell; else over the 27 cells).  -1: revert.
template <int G>
__device__ int group_surface_choice(const MeshView &M, const AsmParams &A, float3 y, int c, float &dist,
                                    const uint2 *pre = nullptr, float *cert_r = nullptr) {
    if (A.cascade) {
        if (c >= 0 && c < A.nt) {
            float d = 0.f;
            const bool on = surface_candidate(M, A, c, y, d);   // every lane, same answer
            if (on) {
                dist = d;
                return c;
            }
        }
        const int t = group_project_surface<G>(M, A, y, dist, true);
        if (t >= 0) return t;
    }
    return group_project_surface<G>(M, A, y, dist, false, pre, A.cascade ? nullptr : cert_r);
}

// distance from y to the faces of the 3 x 3 x 3 triangle-cell block around
// its cell (0 when y lies outside the grid): no triangle outside the block
// comes closer than this
__device__ inline float block_margin(const AsmParams &A, float3 y) {
    const float v[3] = {y.x, y.y, y.z};
    float m = FLT_MAX;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float t = __fmul_rn(__fsub_rn(v[k], A.tg_o[k]), A.tg_inv);
        const float c = (float)cell_coord(v[k], A.tg_o[k], A.tg_inv, A.tg_n[k]);
        m = fminf(m, fminf(t - (c - 1.f), (c + 2.f) - t));
    }
    return fmaxf(m, 0.f) / A.tg_inv;
}

// Closest-feature sign (reading: closest point over the 27 triangle cells,
// sign of the angle-weighted pseudonormal): 1 inside, 0 outside, -1 when no
// triangle lies in range.  *clear gets a lower bound of the distance from y
// to the surface, valid when inside.
template <int G>
__device__ int group_closest_sign(const MeshView &M, const AsmParams &A, float3 y, float &clear,
                                  const uint2 *pre = nullptr) {
    float best = FLT_MAX;
    int bt = 0x7fffffff, breg = 0;
    float3 bcp = make_float3(0.f, 0.f, 0.f);
    for_27_candidates<G>(M, A, y, false, [&](int t) {
        const size_t g = (size_t)(A.tri_off + t);
        const float3 n = f3(M.geo[5 * g + 1]);
        if (n.x == 0.f && n.y == 0.f && n.z == 0.f) return;   // degenerate
        int reg;
        const float3 cp = closest_on_triangle(y, f3(M.vx[3 * g]), f3(M.vx[3 * g + 1]), f3(M.vx[3 * g + 2]), reg);
        const float3 w = y - cp;
        const float dd = dot3(w, w);
        if (dd < best || (dd == best && t < bt)) {
            best = dd;
            bt = t;
            breg = reg;
            bcp = cp;
        }
    }, pre);
    float v = best;
    int t = bt;
    group_argmin<G>(v, t);
    const float blk = block_margin(A, y);
    clear = fmaxf(fminf(t == 0x7fffffff ? FLT_MAX : sqrtf(v), blk) * (1.f - 0x1p-10f) - A.dx * 0x1p-16f, 0.f);
    if (t == 0x7fffffff) return -1;
    // the sign from a lane that holds the winner
    int src = (int)(threadIdx.x & 31u);
    if (G > 1) src = __ffs(__ballot_sync(group_mask<G>(), bt == t && best == v) & group_mask<G>()) - 1;
    int inside = 0;
    if ((int)(threadIdx.x & 31u) == src) {
        const size_t g = (size_t)(A.tri_off + bt);
        const float3 psi = breg == 0 ? f3(M.geo[5 * g + 1]) : f3(M.pn[6 * g + breg - 1]);
        inside = dot3(y - bcp, psi) <= 0.f;
    }
    return G > 1 ? __shfl_sync(group_mask<G>(), inside, src) : inside;
}

// Volume test of a particle of the body: the closest-feature sign, inside
// when no triangle is in range (a step is below a cell)
template <int G>
__device__ inline bool group_volume_inside(const MeshView &M, const AsmParams &A, float3 y, float &clear,
                                           const uint2 *pre = nullptr) {
    return group_closest_sign<G>(M, A, y, clear, pre) != 0;
}

// Boolean partner rule (1 stay outside, 2 stay inside, 0 none) for point x:
// with no partner triangle in range the particle is where it started
template <int G>
__device__ inline bool group_partner_ok(const MeshView &M, const AsmParams &Q, int rule, float3 x) {
    if (rule == 0) return true;
    float unused;
    const int t = group_closest_sign<G>(M, Q, x, unused);
    return rule == 1 ? t != 1 : t != 0;
}

// the segments [x, y) a feature particle projects onto: its own line's, all of
// the body's when it has none yet
__device__ inline int2 line_segments(const MeshView &M, const AsmParams &A, int cons) {
    if (cons < 0 || cons >= A.nseg) return make_int2(0, max(A.nseg, 0));
    const int line = __float_as_int(M.seg[3 * (size_t)(A.seg_off + cons)].w);
    const int2 L = M.lines[A.line_off + line];
    return make_int2(L.x, L.x + L.y);
}

// the closest point of segments r.x + first, r.x + first + step, ..: best
// squared distance, segment (ties to the lower one; -1 for none) and point
__device__ inline void closest_on_segments(const float4 *seg, int seg_off, float3 y, int2 r, int first, int step,
                                           float &best, int &bs, float3 &bq) {
    best = FLT_MAX;
    bs = -1;
    bq = y;
    for (int s = r.x + first; s < r.y; s += step) {
        const float4 *sg = seg + 3 * (size_t)(seg_off + s);
        const float3 a = f3(sg[0]), e = f3(sg[1]) - a;
        const float ee = dot3(e, e);
        float t = ee > 0.f ? dot3(y - a, e) / ee : 0.f;
        t = fminf(fmaxf(t, 0.f), 1.f);
        const float3 q = a + t * e;
        const float3 w = y - q;
        const float dd = dot3(w, w);
        if (dd < best) {
            best = dd;
            bs = s;
            bq = q;
        }
    }
}

// the same over a group of G lanes that hold the same y and r: every lane
// gets the closest of all
template <int G>
__device__ bool group_project_feature(const float4 *segs, int seg_off, float3 y, int2 r, float3 &x, int &seg) {
    float best;
    closest_on_segments(segs, seg_off, y, r, group_lane<G>(), G, best, seg, x);
    if (G > 1) {
        float v = best;
        int t = seg < 0 ? 0x7fffffff : seg;
        const int mine = t;
        group_argmin<G>(v, t);
        const uint32_t own = __ballot_sync(group_mask<G>(), mine == t) & group_mask<G>();
        const int src = __ffs(own) - 1;     // (none anywhere: every lane, with its y)
        x.x = __shfl_sync(group_mask<G>(), x.x, src);
        x.y = __shfl_sync(group_mask<G>(), x.y, src);
        x.z = __shfl_sync(group_mask<G>(), x.z, src);
        seg = t == 0x7fffffff ? -1 : t;
    }
    return seg >= 0;
}

// some triangle of body Q within the 27 triangle cells of x (its dilated
// occupancy bit)
__device__ inline bool near_body(const MeshView &M, const AsmParams &Q, float3 x) {
    return test_bit(M.occ, Q.dil_off,
                    tri_key(Q, cell_coord(x.x, Q.tg_o[0], Q.tg_inv, Q.tg_n[0]),
                            cell_coord(x.y, Q.tg_o[1], Q.tg_inv, Q.tg_n[1]),
                            cell_coord(x.z, Q.tg_o[2], Q.tg_inv, Q.tg_n[2])));
}

// segments of a feature line that the step walks itself.  Cylinder of 105 k
// particles, step and search together with its lines in the step / the search:
// lines of 4 segments 20.2 / 20.6 us, 24 23.8 / 20.6, 64 35.2 / 22.1, 128 54.6 / 24.7.
constexpr int kLaneSegments = 8;

// ---- A5 + A6 -------------------------------------------------------------------
// k_step: one thread per particle (key order): the limited step and its
// tangential part, then the cases that need no search -- feature particles
// of short lines, volume particles with no triangle in the 27
// cells (accepted), surface particles with none (reverted).  Every other
// particle is queued with its trial point for k_search.
__global__ void __launch_bounds__(TPB, 5) k_step(const float4 *__restrict__ pos_s, const float4 *__restrict__ acc_s,
                                              const uint32_t *__restrict__ id_s, int64_t N,
                                              const AsmParams *__restrict__ P, const uint32_t *__restrict__ amax,
                                              float4 *__restrict__ pos, int32_t *__restrict__ cons, MeshView M,
                                              uint32_t *__restrict__ maxdisp, int4 *__restrict__ work,
                                              uint2 *__restrict__ work_r, uint32_t *__restrict__ work_count,
                                              const float4 *__restrict__ cert, const int32_t *__restrict__ cons_s) {
    const int64_t k = (int64_t)blockIdx.x * TPB + threadIdx.x;
    const bool active = k < N;
    // the particle's streams are read together, before its class is known
    // (one round trip to memory instead of two)
    const float4 p = active ? pos_s[k] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 a = active ? acc_s[k] : make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t i = active ? id_s[k] : 0u;
    const int c = active ? cons_s[k] : -1;
    const int cls = active ? cls_of(p.w) : kClsI;
    const int b = active ? body_of(p.w) : 0;
    const AsmParams &A = P[b];
    float disp = 0.f;
    bool queue = false;
    uint2 rng = make_uint2(0u, 0u);   // candidate list of the trial point's triangle cell
    float3 y = f3(p);
    if (active && is_mobile(cls, A) && !is_ghost(p.w)) {
        const float am = __uint_as_float(amax[A.amax_slot]);
        const float sc = am > 0.f ? A.step_h / am : 0.f;     // dt^2 with dt = 0.25 sqrt(h / amax)
        float3 dr = make_float3(a.x * sc, a.y * sc, a.z * sc);
        if (cls == kClsS && c >= 0 && c < A.nt) {
            const float3 n = f3(M.geo[5 * (size_t)(A.tri_off + c) + 1]);
            dr = dr - dot3(dr, n) * n;
        } else if (cls == kClsF && c >= 0 && c < A.nseg) {
            const float3 tau = f3(M.seg[3 * (size_t)(A.seg_off + c) + 2]);
            dr = dot3(dr, tau) * tau;
        }
        const float3 p3 = f3(p);
        y = p3 + dr;
        if (cls == kClsF) {
            // a long line goes to the search, whose lanes share its segments
            // (one lane on a rim of 240 segments kept its warp here for over
            // 10,000 instructions: the step of the gear, 2.4 M particles,
            // 142 -> 76 us, its search 21 -> 37)
            const int2 line = line_segments(M, A, c);
            float3 x;
            int cn = -1;
            float best;
            if (line.y - line.x > kLaneSegments) queue = true;
            else closest_on_segments(M.seg, A.seg_off, y, line, 0, 1, best, cn, x);
            if (cn >= 0) {
                // a partner's triangles within reach: the search tests that
                // partner's rule on the projection (a particle on the
                // intersection curve with a partner lies on both surfaces:
                // no rule of that partner)
                bool near_partner = false;
                for (int q = 0; q < A.npart && !near_partner; q++)
                    if (A.partner_surf[q] != 0 && !(cn >= A.curve_lo[q] && cn < A.curve_hi[q]))
                        near_partner = near_body(M, P[A.partner[q]], x);
                if (near_partner) {
                    queue = true;
                } else {
                    pos[i] = make_float4(x.x, x.y, x.z, p.w);
                    cons[i] = cn;
                    const float3 w = x - p3;
                    disp = sqrtf(dot3(w, w));
                }
            }
        } else {
            const int cx = cell_coord(y.x, A.tg_o[0], A.tg_inv, A.tg_n[0]);
            const int cy = cell_coord(y.y, A.tg_o[1], A.tg_inv, A.tg_n[1]);
            const int cz = cell_coord(y.z, A.tg_o[2], A.tg_inv, A.tg_n[2]);
            bool certified = false;
            bool near_partner = false;
            // some triangle of the body within the 27 triangle cells of y
            const bool near_own = test_bit(M.occ, A.dil_off, tri_key(A, cx, cy, cz));
            if (cls == kClsV && A.vol_rules) {
                for (int q = 0; q < A.npart && !near_partner; q++)
                    if (A.partner_vol[q] != 0) near_partner = near_body(M, P[A.partner[q]], y);
            } else if (cls == kClsV && A.closed && near_own) {
                // (with no triangle near, the volume test accepts anyway: the
                // certificate is not read)
                // inside a ball that an earlier search found free of surface
                // and inside the body: the volume test would accept
                const float4 cc = cert[i];
                const float3 w = y - f3(cc);
                certified = cc.w > 0.f && sqrtf(dot3(w, w)) + cc.w * 0x1p-6f + A.dx * 0x1p-10f < cc.w;
            }
            bool surf_cert = false;
            float3 xs = y;
            if (cls == kClsS && c >= 0 && c < A.nt && !A.cascade) {
                // inside a ball where an earlier search found exactly one
                // projectable candidate of the same triangle cell: the own
                // triangle is the choice when it is projectable here, and lies
                // this close (so it is a candidate of this cell); with no
                // Boolean partner's triangle near the foot the partner rules
                // hold as they would in the search
                const float4 cc = cert[i];
                const float3 w = y - f3(cc);
                if (cc.w < 0.f && sqrtf(dot3(w, w)) < -cc.w &&
                    tri_key(A, cell_coord(cc.x, A.tg_o[0], A.tg_inv, A.tg_n[0]),
                            cell_coord(cc.y, A.tg_o[1], A.tg_inv, A.tg_n[1]),
                            cell_coord(cc.z, A.tg_o[2], A.tg_inv, A.tg_n[2])) == tri_key(A, cx, cy, cz)) {
                    float d;
                    if (surface_candidate(M, A, c, y, d) && fabsf(d) <= A.dx * 0x1p-10f) {
                        surf_cert = true;
                        xs = y - d * f3(M.geo[5 * (size_t)(A.tri_off + c) + 1]);
                        for (int q = 0; q < A.npart && surf_cert; q++)
                            if (A.partner_surf[q] != 0 && near_body(M, P[A.partner[q]], xs)) surf_cert = false;
                    }
                }
            }
            if (certified) {
                pos[i] = make_float4(y.x, y.y, y.z, p.w);
                disp = sqrtf(dot3(dr, dr));
            } else if (surf_cert) {
                pos[i] = make_float4(xs.x, xs.y, xs.z, p.w);
                const float3 w = xs - p3;
                disp = sqrtf(dot3(w, w));
            } else if (near_partner || near_own) {
                queue = true;
                rng = cand_range(M, A, tri_key(A, cx, cy, cz));
            } else if (cls == kClsV) {       // nothing near: inside, accept
                pos[i] = make_float4(y.x, y.y, y.z, p.w);
                disp = sqrtf(dot3(dr, dr));
            }                                // S with nothing near: revert
        }
    }
    // warp-aggregated append to the search queue: surface and feature
    // particles from the front (count work_count[0]), volume particles from
    // the back (work_count[1]), so that a warp of the thread-per-particle
    // search meets one kind of test
    const bool qv = queue && cls == kClsV, qs = queue && cls != kClsV;
    const uint32_t ms = __ballot_sync(0xffffffffu, qs), mv = __ballot_sync(0xffffffffu, qv);
    if (ms | mv) {
        const int lane = threadIdx.x & 31;
        const int ls = ms ? __ffs(ms) - 1 : 0, lv = mv ? __ffs(mv) - 1 : 0;
        uint32_t bs = 0u, bv = 0u;
        if (ms && lane == ls) bs = atomicAdd(work_count, (uint32_t)__popc(ms));
        if (mv && lane == lv) bv = atomicAdd(work_count + 1, (uint32_t)__popc(mv));
        bs = __shfl_sync(0xffffffffu, bs, ls);
        bv = __shfl_sync(0xffffffffu, bv, lv);
        const int4 it = make_int4((int)k, __float_as_int(y.x), __float_as_int(y.y), __float_as_int(y.z));
        if (qs) {
            const uint32_t q = bs + __popc(ms & lanemask_lt());
            if (FPPG_CHECK(q < N, kChkQueue)) {
                work[q] = it;
                work_r[q] = rng;
            }
        }
        if (qv) {
            const int64_t q = N - 1 - (int64_t)(bv + __popc(mv & lanemask_lt()));
            if (FPPG_CHECK(q >= 0 && q < N, kChkQueue)) {
                work[q] = it;
                work_r[q] = rng;
            }
        }
    }
    __shared__ int s_lab[TPB / 32];
    __shared__ uint32_t s_max[TPB / 32];
    block_labelled_max<TPB / 32>(maxdisp, b, disp, s_lab, s_max);
}

// entry e of the two-ended search queue: the nf front entries first, then
// the back ones from slot N - 1 downwards
__device__ inline int64_t queue_slot(uint32_t nf, int64_t N, uint32_t e) {
    return e < nf ? (int64_t)e : N - 1 - (int64_t)(e - nf);
}


// k_search: G lanes per queued particle (grid-stride over the queue): surface
// particles go to the closest projectable triangle or revert, volume particles
// are accepted when the pseudonormal sign says inside.  Bound by the latency of
// its dependent loads, so what counts is how many particles are in flight and
// how many of a group's lanes the candidate list feeds (lists of 4.7 on the gear:
// 39.8 us an iteration with 8 lanes, 54.8 with 32; Group::set_search_lanes).
// At most 64 registers (four blocks, 32 warps per SM).
template <int G>
__global__ void __launch_bounds__(TPB, 4) k_search(const float4 *__restrict__ pos_s,
                                                   const uint32_t *__restrict__ id_s,
                                                   const AsmParams *__restrict__ P, float4 *__restrict__ pos,
                                                   int32_t *__restrict__ cons, MeshView M,
                                                   uint32_t *__restrict__ maxdisp, const int4 *__restrict__ work,
                                                   const uint2 *__restrict__ work_r,
                                                   const uint32_t *__restrict__ work_count, int64_t N,
                                                   float4 *__restrict__ cert) {
    const uint32_t nf = work_count[0], n = nf + work_count[1];
    const uint32_t stride = gridDim.x * (TPB / G);
    const bool lead = group_lane<G>() == 0;
    // the leader's running max move of body run_b, added when the body
    // changes and once at the end (the queue is in key order: few changes)
    int run_b = 0;
    float run = 0.f;
    for (uint32_t e = (blockIdx.x * TPB + threadIdx.x) / G; e < n; e += stride) {
        const int64_t qs = queue_slot(nf, N, e);
        if (!FPPG_CHECK(qs >= 0 && qs < N, kChkQueue)) continue;
        const int4 it = work[qs];
        const uint2 rng = work_r[qs];
        if (!FPPG_CHECK(it.x >= 0 && it.x < N, kChkEntry)) continue;
        const float3 y = make_float3(__int_as_float(it.y), __int_as_float(it.z), __int_as_float(it.w));
        const float4 p = pos_s[it.x];
        const uint32_t i = id_s[it.x];
        const int cls = cls_of(p.w), b = body_of(p.w);
        const AsmParams &A = P[b];
        float3 x = y;
        int tri = -2;
        float clear = 0.f;
        bool ok;
        if (cls == kClsS) {
            float d;
            tri = group_surface_choice<G>(M, A, y, A.cascade ? cons[i] : -1, d, &rng, &clear);
            ok = tri >= 0;
            if (ok) x = y - d * f3(M.geo[5 * (size_t)(A.tri_off + tri) + 1]);
        } else if (cls == kClsF) {
            // a feature particle of a long line, or of a union member near
            // the partner: its projection (again), then the partner test below
            ok = group_project_feature<G>(M.seg, A.seg_off, y, line_segments(M, A, cons[i]), x, tri);
        } else {
            ok = group_volume_inside<G>(M, A, y, clear, &rng);
        }
        // Boolean operations: the partner rule of the particle's class
        for (int q = 0; q < A.npart && ok; q++)
            if (!(cls == kClsF && tri >= A.curve_lo[q] && tri < A.curve_hi[q]))
                ok = group_partner_ok<G>(M, P[A.partner[q]], cls == kClsV ? A.partner_vol[q] : A.partner_surf[q], x);
        if (G > 1) __syncwarp(group_mask<G>());   // (cons[i] is read by every lane of the group above)
        if (ok && lead) {
            pos[i] = make_float4(x.x, x.y, x.z, p.w);
            if (tri >= 0) cons[i] = tri;
            if (cls == kClsV && A.closed && !A.vol_rules) cert[i] = make_float4(y.x, y.y, y.z, clear);
            // surface certificates carry a negative radius (never taken for an inside one)
            if (cls == kClsS && clear > 0.f) cert[i] = make_float4(y.x, y.y, y.z, -clear);
            const float3 w = x - f3(p);
            if (b != run_b) {
                if (run > 0.f) atomicMax(maxdisp + run_b, __float_as_uint(run));
                run_b = b;
                run = 0.f;
            }
            run = fmaxf(run, sqrtf(dot3(w, w)));
        }
    }
    __syncwarp();
    labelled_max(maxdisp, run_b, run);
}

// ---- diagnostics --------------------------------------------------------------
__global__ void k_unpermute(const float4 *__restrict__ acc_s, const uint32_t *__restrict__ id_s, int64_t N,
                            float *__restrict__ acc, const int32_t *__restrict__ cnt_s, int32_t *__restrict__ cnt) {
    int64_t k = (int64_t)blockIdx.x * TPB + threadIdx.x;
    if (k >= N) return;
    uint32_t i = id_s[k];
    if (acc) {
        float4 a = acc_s[k];
        acc[3 * (size_t)i] = a.x;
        acc[3 * (size_t)i + 1] = a.y;
        acc[3 * (size_t)i + 2] = a.z;
    }
    if (cnt) cnt[i] = cnt_s[k];
}

__global__ void k_project_points(const float *__restrict__ y, const int32_t *__restrict__ cls,
                                  const int32_t *__restrict__ cons_in, int64_t n, const AsmParams *__restrict__ P,
                                  MeshView M, float *__restrict__ x, int32_t *__restrict__ cons_out,
                                  int32_t *__restrict__ ok) {
    const int64_t i = ((int64_t)blockIdx.x * TPB + threadIdx.x) / 32;   // one warp per point
    const int lane = threadIdx.x & 31;
    if (i >= n) return;                                                    // whole warp
    const AsmParams &A = P[0];
    const float3 yy = make_float3(y[3 * i], y[3 * i + 1], y[3 * i + 2]);
    float3 xx = yy;
    const int c = cons_in ? cons_in[i] : -1;
    int cn = c;
    bool r = true;
    const int cl = cls[i];
    if (cl == kClsS) {
        float d;
        const int t = group_surface_choice<32>(M, A, yy, c, d);
        r = t >= 0;
        if (r) {
            xx = yy - d * f3(M.geo[5 * (size_t)(A.tri_off + t) + 1]);
            cn = t;
        }
    } else if (cl == kClsV) {
        float clear;
        r = group_volume_inside<32>(M, A, yy, clear);
    } else if (cl == kClsF) {
        r = group_project_feature<32>(M.seg, A.seg_off, yy, line_segments(M, A, c), xx, cn);
    }
    if (!r) {
        xx = yy;
        cn = c;
    }
    if (lane == 0) {
        x[3 * i] = xx.x;
        x[3 * i + 1] = xx.y;
        x[3 * i + 2] = xx.z;
        cons_out[i] = cn;
        ok[i] = r ? 1 : 0;
    }
}

} // namespace

// ---- host driver ----------------------------------------------------------------
// A1-A3 of the counted form: key[0] the keys and id[0] the arrival places by
// id, id[1] the ids in arrival order, key[1] the ids in key order
static void build_counted(DevGroup &d, cudaStream_t s) {
    const int64_t F1 = kSlabs * d.total_cells + 1, nt = count_tiles(F1);
    k_keys_count<<<nblocks(d.N), TPB, 0, s>>>(d.pos, d.N, d.params, d.key[0], d.id[0], d.cnt, F1 - 1);
    const uint32_t *tiles = nullptr;
    if (nt > kFewTiles) {
        k_tile_sums<<<(unsigned)nt, TPB, 0, s>>>(d.cnt, F1, d.tiles);
        tiles = d.tiles;
    }
    if (nt > kScanTiles) {
        exclusive_scan_u32(d.tiles, d.tile_base, nt, nullptr, d.scan_tmp, scan_tmp_elems(nt), s);
        tiles = d.tile_base;
    }
    k_count_starts<<<(unsigned)nt, TPB, 0, s>>>(d.cnt, tiles, nt > kScanTiles, F1, d.fstart, d.amax, d.maxdisp, d.B,
                                                d.work_count);
    d.id_s = d.key[1];
    // a block for every 4096 counts to clear, however few the particles: 100 of
    // them on 71 M fine keys 4,392 -> 201 us an iteration, on 3.9 M 273 -> 37
    // (radix form 377 and 79)
    k_place<<<std::max(nblocks(d.N), nblocks(F1, kCountTile)), TPB, 0, s>>>(d.key[0], d.id[0], d.fstart, d.N, d.id[1],
                                                                            d.cnt, F1);
    if (d.N < kGatherTwoMinN)
        k_rank_gather<1><<<nblocks(d.N), TPB, 0, s>>>(d.id[1], d.params, d.fstart, d.pos, d.cons, d.N, d.pos_s,
                                                      d.pos_p, d.id_s, d.cons_s, F1 - 1);
    else
        k_rank_gather<2><<<nblocks(d.N, 2 * TPB), TPB, 0, s>>>(d.id[1], d.params, d.fstart, d.pos, d.cons, d.N,
                                                               d.pos_s, d.pos_p, d.id_s, d.cons_s, F1 - 1);
}

uint32_t *Group::count_crowds(int64_t n, cudaStream_t s) {
    const int64_t F1 = kSlabs * d.total_cells + 1;
    cudaMemsetAsync(d.totals, 0, sizeof(uint32_t), s);
    k_crowd_counts<<<nblocks(n), TPB, 0, s>>>(d.pos, n, d.params, d.cnt, F1 - 1);
    k_crowd_max<<<std::min<unsigned>(nblocks(F1, 16 * TPB), 152 * 8), TPB, 0, s>>>(d.cnt, F1, d.totals);
    return d.totals;
}

int Group::find_crowds(cudaStream_t s, bool *found, std::string &err) {
    uint32_t most = 0u;
    cudaError_t e = cudaSuccess;
    if (d.N > kCrowd) {
        // (the counters may be at work in a relaxation on a stream that the
        // caller has left)
        e = cudaDeviceSynchronize();
        if (e == cudaSuccess) count_crowds(d.N, s);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&most, d.totals, sizeof(most), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
    if (e != cudaSuccess) {
        err = std::string("crowded keys: ") + cudaGetErrorString(e);
        return 4;
    }
    *found = most > kCrowd;
    return 0;
}

void build_grid_dev(DevGroup &d, cudaStream_t s) {
    if (d.counted) {
        build_counted(d, s);
        return;
    }
    k_keys<<<nblocks(std::max<int64_t>(d.N, d.B)), TPB, 0, s>>>(d.pos, d.N, d.params, d.key[0], d.amax, d.maxdisp, d.B,
                                                                 d.work_count);
    const int buf = radix_sort_u32(d.key, d.id, true, d.N, d.key_bits, d.hist, d.totals, s);
    d.id_s = d.id[buf];
    d.key_s = d.key[buf];
    k_gather<<<nblocks(d.N), TPB, 0, s>>>(d.id_s, d.pos, d.N, d.pos_s, d.pos_p, d.cons, d.cons_s);
    // the start table from the sorted keys
    const int64_t F1 = kSlabs * d.total_cells + 1;
    const int64_t nblk = start_blocks(F1);
    k_key_block_starts<<<nblocks(d.N + 1), TPB, 0, s>>>(d.key_s, d.N, nblk, d.bstart);
    k_fine_starts<<<(unsigned)nblk, kStartBlock, 0, s>>>(d.key_s, d.bstart, F1, d.fstart);
}

const uint32_t *sorted_keys(DevGroup &d, cudaStream_t s) {
    if (!d.counted) return d.key_s;
    k_sorted_keys<<<nblocks(d.N), TPB, 0, s>>>(d.id_s, d.key[0], d.N, d.id[1]);   // the arrival order is used up
    return d.id[1];
}

int grid_kernels(const DevGroup &d) {
    if (!d.counted) return 1 + 3 * d.passes + 3;   // keys, radix passes, gather, block starts, fine-key starts
    const int64_t nt = count_tiles(kSlabs * d.total_cells + 1);
    return 4 + (nt > kFewTiles ? 1 : 0) + (nt > kScanTiles ? scan_launches(nt) : 0);
}

void build_grid(Group &g, cudaStream_t s) { build_grid_dev(g.d, s); }

void forces_dev(DevGroup &d, int tb, int variant, cudaStream_t s, int32_t *count_s, int32_t *tested_s) {
    const bool split = !count_s && variant == 0 && d.N <= kSplitMaxN;
    const unsigned nbk = nblocks(d.N, split ? tb / 2 : tb);
#define FPPG_FORCE(V, C, M, S)                                                                                       \
    k_force<V, C, M, S><<<nbk, tb, 0, s>>>(d.pos_s, d.pos_p, d.N, d.params, d.fstart, d.acc_s, d.amax, count_s,       \
                                           tested_s)
#define FPPG_FORCE_ORDER(V, C, S)                                                                                    \
    do {                                                                                                             \
        if (d.morton_rows) FPPG_FORCE(V, C, true, S);                                                                \
        else FPPG_FORCE(V, C, false, S);                                                                             \
    } while (0)
    if (split) FPPG_FORCE_ORDER(0, false, true);
    else if (count_s && variant == 1) FPPG_FORCE_ORDER(1, true, false);
    else if (count_s) FPPG_FORCE_ORDER(0, true, false);
    else if (variant == 1) FPPG_FORCE_ORDER(1, false, false);
    else FPPG_FORCE_ORDER(0, false, false);
#undef FPPG_FORCE_ORDER
#undef FPPG_FORCE
}

void forces(Group &g, cudaStream_t s, int32_t *count_s, int32_t *cand_s, int32_t *tested_s) {
    DevGroup &d = g.d;
    forces_dev(d, g.force_block, g.force_variant, s, count_s, tested_s);
    if (cand_s)
        k_count<<<nblocks(d.N), TPB, 0, s>>>(d.pos_s, d.N, d.params, d.fstart, nullptr, cand_s);
}

static void search(Group &g, cudaStream_t s) {
    DevGroup &d = g.d;
#define FPPG_SEARCH(G)                                                                                               \
    k_search<G><<<g.search_blocks, TPB, 0, s>>>(d.pos_s, d.id_s, d.params, d.pos, d.cons, g.mesh, d.maxdisp, d.work,  \
                                                queue_ranges(d), d.work_count, d.N, d.cert)
    if (g.search_thread) FPPG_SEARCH(1);
    else if (g.search_lanes == 8) FPPG_SEARCH(8);
    else FPPG_SEARCH(32);
#undef FPPG_SEARCH
}

void iterate(Group &g, cudaStream_t s, bool energy_mode, int32_t *count_dbg) {
    DevGroup &d = g.d;
    if (d.N == 0) return;
    // phase timing: events before A1, after A3, after A4, after A5 and after A6
    const bool timed = g.time_force && g.ev_used + kPhaseEvents <= (int)g.ev.size();
    // inside a stream capture the records must be external so that they
    // become event-record nodes whose timestamps can be read after a replay
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (timed) cudaStreamIsCapturing(s, &cap);
    const unsigned flags = cap == cudaStreamCaptureStatusActive ? cudaEventRecordExternal : 0u;
    if (timed) cudaEventRecordWithFlags(g.ev[g.ev_used], s, flags);
    {
        NvtxRange r("A1-A3 grid");
        build_grid(g, s);
    }
    if (timed) cudaEventRecordWithFlags(g.ev[g.ev_used + 1], s, flags);
    {
        NvtxRange r("A4 force");
        if (energy_mode) energy_accel(g, s);
        else forces(g, s, count_dbg);
    }
    if (timed) cudaEventRecordWithFlags(g.ev[g.ev_used + 2], s, flags);
    NvtxRange r("A5-A6 step and search");
    k_step<<<nblocks(d.N), TPB, 0, s>>>(d.pos_s, d.acc_s, d.id_s, d.N, d.params, d.amax, d.pos, d.cons, g.mesh,
                                         d.maxdisp, d.work, queue_ranges(d), d.work_count, d.cert, d.cons_s);
    if (timed) cudaEventRecordWithFlags(g.ev[g.ev_used + 3], s, flags);
    search(g, s);
    if (timed) {
        cudaEventRecordWithFlags(g.ev[g.ev_used + 4], s, flags);
        g.ev_used += kPhaseEvents;
    }
}

void step_and_project(Group &g, cudaStream_t s) {
    DevGroup &d = g.d;
    if (d.N == 0) return;
    k_step<<<nblocks(d.N), TPB, 0, s>>>(d.pos_s, d.acc_s, d.id_s, d.N, d.params, d.amax, d.pos, d.cons, g.mesh,
                                         d.maxdisp, d.work, queue_ranges(d), d.work_count, d.cert, d.cons_s);
    search(g, s);
}

namespace {
__global__ void k_tag_ghosts(float4 *__restrict__ pos, int64_t n, int64_t first_ghost) {
    const int64_t i = (int64_t)blockIdx.x * TPB + threadIdx.x;
    if (i >= n) return;
    const uint32_t w = __float_as_uint(pos[i].w);
    pos[i].w = __uint_as_float(i >= first_ghost ? (w | kGhostBit) : (w & ~kGhostBit));
}
} // namespace

void tag_ghosts(Group &g, int64_t first_ghost, cudaStream_t s) {
    if (g.d.N > 0) k_tag_ghosts<<<nblocks(g.d.N), TPB, 0, s>>>(g.d.pos, g.d.N, first_ghost);
}

void unpermute_dev(DevGroup &d, cudaStream_t s, float *acc_out, const int32_t *count_s,
                   int32_t *count_out) {
    k_unpermute<<<nblocks(d.N), TPB, 0, s>>>(d.acc_s, d.id_s, d.N, acc_out, count_s, count_out);
}

void unpermute(Group &g, cudaStream_t s, float *acc_out, const int32_t *count_s, int32_t *count_out) {
    unpermute_dev(g.d, s, acc_out, count_s, count_out);
}

void project_points(Group &g, const float *y, const int32_t *cls, const int32_t *cons_in, int64_t n, float *x,
                    int32_t *cons_out, int32_t *ok, cudaStream_t s) {
    k_project_points<<<nblocks(32 * n), TPB, 0, s>>>(y, cls, cons_in, n, g.d.params, g.mesh, x, cons_out, ok);
}

} // namespace fppg
