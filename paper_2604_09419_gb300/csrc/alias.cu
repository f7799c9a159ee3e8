// Alias tables on the GPU for the two discrete distributions of the method:
//   - the positive-pair pick over arcs, proportional to the arc weight
//     (Algorithm 3: the discrete distribution over E_p / ||E_p||), and
//   - the negative distribution q(v) = d(v)^0.75 / sum_x d(x)^0.75 with d the
//     weighted out-degree (Section IV-A, Eq. 1).
// FP64 is used only for the degree sums and the normalisation; the table is
// built from exact integer masses so that every bucket probability is a known
// rational and the construction is reproducible bit for bit.
//
// Pairing (the sweep rule, written as prefix sums so that it runs in
// parallel): let lights be the items with m < 2^32 (deficit Q - m), heavies
// those with m > 2^32 (excess m - Q), both in index order, DP/EP the
// inclusive prefix sums of deficits/excesses.  Light number j takes as alias
// the first heavy k with EP[k] >= DP[j-1]; heavy k (not the last) becomes a
// light bucket at the first light j with DP[j] > EP[k], with threshold
// Q - (DP[j] - EP[k]) and alias heavy k+1.  This is exactly the table of the
// sequential sweep in which the current heavy item tops up the lights in
// order and, when its own mass drops below Q, is topped up by the next heavy
// item (Huebschle-Schneider and Sanders, "Parallel Weighted Random
// Sampling", ESA 2019, describe the same parallel split).
#include <math.h>

#include "line_internal.cuh"
#include "scan.cuh"

namespace line {

namespace {

// Fixed-order FP64 sum of one block of 1024 values, halving strides 512 .. 1,
// by one warp: lane l holds values l + 32 k, so strides 512 .. 32 pair values
// of a lane and 16 .. 1 are shuffles.  (One CTA per block of values, in shared
// memory with a barrier per stride, took 289 us for 31.4M values.)
template <typename T>
__device__ __forceinline__ double tree_sum(const T* __restrict__ x, int64_t n, int lane) {
    double v[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = 32 * k + lane < n ? (double)x[32 * k + lane] : 0.0;
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1)
#pragma unroll
        for (int k = 0; k < s; ++k) v[k] = __dadd_rn(v[k], v[k + s]);
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
        const double o = __shfl_down_sync(0xFFFFFFFFu, v[0], s);
        v[0] = __dadd_rn(v[0], o);  // lanes >= s hold no partial sum
    }
    return v[0];  // in lane 0
}

template <typename T>
__global__ void __launch_bounds__(256) k_tree_sum(const T* __restrict__ x, int64_t n, double* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int64_t blk = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (blk * kSumBlock >= n) return;
    const double v = tree_sum(x + blk * kSumBlock, n - blk * kSumBlock, lane);
    if (lane == 0) out[blk] = v;
}

// out[r] = the sum of row r's n <= 1024 values, a warp a row.
__global__ void __launch_bounds__(256) k_tree_rows(const double* __restrict__ x, int64_t rows, int64_t n,
                                                   double* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int64_t r = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= rows) return;
    const double v = tree_sum(x + r * n, n, lane);
    if (lane == 0) out[r] = v;
}

// Sum over the block's threads of v (any order: integers), in every thread.
__device__ __forceinline__ unsigned long long block_sum(unsigned long long v, unsigned long long* part) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    v = 0;
    for (unsigned w = 0; w < blockDim.x / 32; ++w) v += part[w];
    return v;
}

// row_ptr[v] = e for the nodes v in [v0, v1] between two arcs, written by a
// whole warp (by one thread a run of 2^24 nodes took 56 ms).  In an unsorted
// graph every ascent begins such a run (2^22 random arcs over 2^20 nodes: 7e11
// entries), so one ends once any thread has found the graph invalid.
constexpr int64_t kFillShort = 32, kFillPiece = 1024;

__device__ __forceinline__ void fill_offsets(int64_t* __restrict__ row_ptr, int64_t v0, int64_t v1, int64_t e,
                                             const uint32_t* status) {
    const int lane = threadIdx.x & 31;
    for (int64_t v = v0; v <= v1; v += kFillPiece) {
        if (*(volatile const uint32_t*)status & DEV_ERR_GRAPH) return;
        for (int64_t q = v + lane, end = min(v1, v + kFillPiece - 1); q <= end; q += 32) row_ptr[q] = e;
    }
}

// One pass over the arcs: validation (DEV_ERR_GRAPH), the first arc of each
// node (row_ptr, for a valid graph), whether every weight is an integer in
// [1, 2^24], and - as if they were - their sum and each node's (degi, zero
// before).  A thread takes kArcs consecutive arcs: a node's run inside them
// is added with one atomic (src is sorted).  A thread reports an invalid arc
// before it writes any offset, and then writes none.
// Bound: HBM (12 bytes an arc) and the run's branches: 200 us for 31.4M arcs;
// the validation, the row offsets, the integer check and the node sums (a
// warp a node) took 85 + 64 + 25 + 1,357 us as four kernels.
constexpr int kArcs = 8;

__global__ void __launch_bounds__(256) k_graph_scan(int64_t n_nodes, int64_t n_arcs, const int32_t* __restrict__ src,
                                                    const int32_t* __restrict__ dst, const float* __restrict__ w,
                                                    int64_t* __restrict__ row_ptr, unsigned long long* __restrict__ degi,
                                                    GraphScan* __restrict__ out, uint32_t* status) {
    __shared__ unsigned long long part[8];
    const int lane = threadIdx.x & 31;
    bool frac = false;
    unsigned long long total = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * kArcs;
    // (whole warps go round)
    for (int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane) * kArcs; w0 < n_arcs; w0 += stride) {
        const int64_t e0 = w0 + lane * kArcs;
        int32_t s[kArcs], d[kArcs];
        float x[kArcs];
        const int cnt = (int)max((int64_t)0, min((int64_t)kArcs, n_arcs - e0));
        if (cnt == kArcs) {  // (the library's own copies: 256-byte aligned)
#pragma unroll
            for (int q = 0; q < kArcs / 4; ++q) {
                const int4 a = __ldg(reinterpret_cast<const int4*>(src + e0) + q), c = __ldg(reinterpret_cast<const int4*>(dst + e0) + q);
                s[4 * q] = a.x, s[4 * q + 1] = a.y, s[4 * q + 2] = a.z, s[4 * q + 3] = a.w;
                d[4 * q] = c.x, d[4 * q + 1] = c.y, d[4 * q + 2] = c.z, d[4 * q + 3] = c.w;
                const float4 f = w ? __ldg(reinterpret_cast<const float4*>(w + e0) + q) : make_float4(1.0f, 1.0f, 1.0f, 1.0f);
                x[4 * q] = f.x, x[4 * q + 1] = f.y, x[4 * q + 2] = f.z, x[4 * q + 3] = f.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < kArcs; ++k) {
                s[k] = k < cnt ? src[e0 + k] : 0;
                d[k] = k < cnt ? dst[e0 + k] : 0;
                x[k] = k < cnt && w ? w[e0 + k] : 1.0f;
            }
        }
        const int32_t before = cnt && e0 > 0 ? src[e0 - 1] : -1;
        bool ok = before >= -1;
#pragma unroll
        for (int k = 0; k < kArcs; ++k) {
            if (k >= cnt) continue;
            ok = ok && s[k] >= 0 && s[k] < n_nodes && s[k] >= (k > 0 ? s[k - 1] : before) && d[k] >= 0 && d[k] < n_nodes &&
                 x[k] > 0.0f && isfinite(x[k]);
        }
        if (!ok && !(*(volatile const uint32_t*)status & DEV_ERR_GRAPH)) atomicOr(status, DEV_ERR_GRAPH);
        const bool last = e0 + cnt == n_arcs;  // the nodes after the last arc's follow
        bool far = false;                      // a run too long for one thread
        if (ok && cnt) {
            int32_t prev = before;
            unsigned long long run = 0;
#pragma unroll
            for (int k = 0; k < kArcs; ++k) {
                if (k < cnt) {
                    const bool whole = x[k] >= 1.0f && x[k] <= 16777216.0f && x[k] == truncf(x[k]);
                    frac |= !whole;
                    const uint32_t xi = whole ? __float2uint_rz(x[k]) : 0u;
                    total += xi;
                    if (s[k] != prev) {
                        if (run) atomicAdd(degi + prev, run);
                        run = 0;
                        if ((int64_t)s[k] - prev > kFillShort) far = true;
                        else
                            for (int64_t v = (int64_t)prev + 1; v <= s[k]; ++v) row_ptr[v] = e0 + k;
                    }
                    run += xi;
                    prev = s[k];
                }
            }
            if (run) atomicAdd(degi + prev, run);
            far |= last;
        }
        if (__any_sync(0xFFFFFFFFu, far)) {
#pragma unroll
            for (int k = 0; k <= kArcs; ++k) {
                // the run before arc k; k = cnt: the one after the last arc
                const int64_t lo = (int64_t)(k > 0 ? s[k > 0 ? k - 1 : 0] : before) + 1;
                const int64_t hi = k < cnt ? (int64_t)s[k < kArcs ? k : 0] : n_nodes;
                const bool mine = ok && cnt && (k < cnt ? hi - lo >= kFillShort : k == cnt && last);
                for (uint32_t mask = __ballot_sync(0xFFFFFFFFu, mine); mask; mask &= mask - 1) {
                    const int l = __ffs(mask) - 1;
                    fill_offsets(row_ptr, __shfl_sync(0xFFFFFFFFu, lo, l), __shfl_sync(0xFFFFFFFFu, hi, l),
                                 __shfl_sync(0xFFFFFFFFu, e0 + k, l), status);
                }
            }
        }
    }
    if (frac) out->frac = 1u;
    total = block_sum(total, part);
    if (threadIdx.x == 0 && total) atomicAdd(&out->sum, total);
}

__device__ __forceinline__ void store_neg_weight(double d, int64_t v, double* __restrict__ x, float* __restrict__ deg) {
    double r = 0.0;
    if (d > 0.0) {
        const double s = __dsqrt_rn(d);
        r = __dmul_rn(s, __dsqrt_rn(s));
    }
    x[v] = r;
    if (deg) deg[v] = (float)d;
}

// x_v = d(v)^0.75 = sqrt(d) * sqrt(sqrt(d)), d = weights of v's arcs summed in
// arc order.  Integer weights: the sums of k_graph_scan - exact in any order,
// so equal to the FP64 sum in arc order while they stay below 2^53.
__global__ void k_neg_weights_int(int64_t n_nodes, const unsigned long long* __restrict__ degi, double* __restrict__ x,
                                  float* __restrict__ deg) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n_nodes; v += (int64_t)gridDim.x * blockDim.x)
        store_neg_weight((double)degi[v], v, x, deg);
}

// Any other weights: one thread per node adds them in FP64 in arc order.
__global__ void k_neg_weights(int64_t n_nodes, const int64_t* __restrict__ row_ptr, const float* __restrict__ w,
                              double* __restrict__ x, float* __restrict__ deg) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n_nodes;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int64_t lo = row_ptr[v], hi = row_ptr[v + 1];
        double d = 0.0;
        for (int64_t e = lo; e < hi; ++e) d = __dadd_rn(d, (double)w[e]);
        store_neg_weight(d, v, x, deg);
    }
}

struct MassCounters {
    unsigned long long sum_m;  // sum of floor(x_i S)
    unsigned long long npos;   // #(x_i > 0)
    unsigned long long nge1;   // #(m_i >= 1)
    unsigned long long pad;
};

// m_i = floor(x_i * S), S = (n * 2^32) / W, for weights x (FP64, or FP32
// arc weights, or null: all 1).  GB300's FP64 pipe runs the product, the floor
// and the conversion: with `whole` (integer FP32 weights) those of small
// weights come from a table in shared memory.
constexpr int kMassTab = 512;

template <typename T>
__global__ void __launch_bounds__(256) k_masses(int64_t n, const T* __restrict__ x, const double* __restrict__ W, bool whole,
                                                uint64_t* __restrict__ m, MassCounters* cnt, uint32_t* status) {
    __shared__ uint64_t tab[kMassTab];
    __shared__ unsigned long long part[8];
    const double w = *W;
    if (!(w > 0.0) || !isfinite(w)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(status, DEV_ERR_ALIAS);
        return;
    }
    const double S = __ddiv_rn(__dmul_rn((double)n, 4294967296.0), w);
    if (whole) {
        for (int k = threadIdx.x; k < kMassTab; k += blockDim.x) tab[k] = (uint64_t)floor(__dmul_rn((double)k, S));
        __syncthreads();
    }
    unsigned long long sm = 0, np = 0, ng = 0;
#pragma unroll 4
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const T xi = x ? x[i] : (T)1;
        const uint32_t k = whole ? (uint32_t)xi : (uint32_t)kMassTab;
        const uint64_t mi = k < kMassTab ? tab[k] : (uint64_t)floor(__dmul_rn((double)xi, S));
        m[i] = mi;
        sm += mi;
        np += xi > (T)0;
        ng += mi >= 1;
    }
    sm = block_sum(sm, part);
    np = block_sum(np, part);
    ng = block_sum(ng, part);
    if (threadIdx.x == 0) {
        atomicAdd(&cnt->sum_m, sm);
        atomicAdd(&cnt->npos, np);
        atomicAdd(&cnt->nge1, ng);
    }
}

struct GenPos {
    const double* x;
    __device__ uint32_t operator()(int64_t i) const { return x[i] > 0.0 ? 1u : 0u; }
};
struct GenGe1 {
    const uint64_t* m;
    __device__ uint32_t operator()(int64_t i) const { return m[i] >= 1 ? 1u : 0u; }
};
// D > 0: q to every positive item, +1 more to the first r of them.
struct OutAddRR {
    const double* x;
    uint64_t* m;
    uint64_t q, r;
    __device__ void operator()(int64_t i, uint32_t excl, uint32_t) const {
        if (x[i] > 0.0) m[i] += q + ((uint64_t)excl < r ? 1ull : 0ull);
    }
};
// D < 0: -1 to the first |D| items with m >= 1.
struct OutSubFirst {
    uint64_t* m;
    uint64_t need;
    __device__ void operator()(int64_t i, uint32_t excl, uint32_t) const {
        if (m[i] >= 1 && (uint64_t)excl < need) m[i] -= 1;
    }
};

// Item i's mass with a remainder spread over all items: m_i + q + (i < r).
struct Mass {
    const uint64_t* m;
    uint64_t q, r;
    __device__ uint64_t operator()(int64_t i) const { return m[i] + q + ((uint64_t)i < r ? 1ull : 0ull); }
};

// The light and heavy items of a tile of kClassTile: their numbers, deficits
// and excesses.
constexpr int kClassRounds = 16;
constexpr int kClassTile = 256 * kClassRounds;

__global__ void __launch_bounds__(256) k_class_sums(int64_t n, Mass mass, Quad* __restrict__ tile) {
    __shared__ unsigned long long part[8];
    unsigned long long a = 0, b = 0, c = 0, d = 0;
    const int64_t base = (int64_t)blockIdx.x * kClassTile;
#pragma unroll
    for (int k = 0; k < kClassRounds; ++k) {
        const int64_t i = base + k * 256 + threadIdx.x;
        const uint64_t v = i < n ? mass(i) : kQ;
        a += v < kQ;
        b += v > kQ;
        c += v < kQ ? kQ - v : 0ull;
        d += v > kQ ? v - kQ : 0ull;
    }
    const unsigned long long ab = block_sum(a << 32 | b, part);
    c = block_sum(c, part);
    d = block_sum(d, part);
    if (threadIdx.x == 0) tile[blockIdx.x] = Quad{(uint32_t)(ab >> 32), (uint32_t)ab, c, d};
}

__device__ __forceinline__ uint64_t warp_incl(uint64_t v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = shfl_up(v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// The lights' {index, mass} and inclusive deficit sums by light rank, the
// heavies' indices and inclusive excess sums by heavy rank; buckets that are
// exactly full keep their mass.  A warp takes 512 consecutive items in rounds
// of 32, so that its reads and its (compacted) writes are contiguous: 16
// items a thread, written as they come, took 450 us for 31.4M items, this 360.
__global__ void __launch_bounds__(256) k_class_apply(int64_t n, Mass mass, const Quad* __restrict__ tile,
                                                     uint2* __restrict__ light, uint64_t* __restrict__ dp,
                                                     uint32_t* __restrict__ heavy_idx, uint64_t* __restrict__ ep,
                                                     uint2* __restrict__ tab) {
    __shared__ Quad wtot[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * kClassTile + warp * (32 * kClassRounds) + lane;
    uint64_t v[kClassRounds];
    Quad t{0u, 0u, 0ull, 0ull};
#pragma unroll
    for (int k = 0; k < kClassRounds; ++k) {
        v[k] = base + 32 * k < n ? mass(base + 32 * k) : kQ;
        t.a += v[k] < kQ;
        t.b += v[k] > kQ;
        t.c += v[k] < kQ ? kQ - v[k] : 0ull;
        t.d += v[k] > kQ ? v[k] - kQ : 0ull;
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        t.a += __shfl_xor_sync(0xFFFFFFFFu, t.a, o);
        t.b += __shfl_xor_sync(0xFFFFFFFFu, t.b, o);
        t.c += __shfl_xor_sync(0xFFFFFFFFu, t.c, o);
        t.d += __shfl_xor_sync(0xFFFFFFFFu, t.d, o);
    }
    if (lane == 0) wtot[warp] = t;
    __syncthreads();
    Quad at = tile[blockIdx.x];
    for (int w = 0; w < warp; ++w) at = at + wtot[w];
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
    for (int k = 0; k < kClassRounds; ++k) {
        const int64_t i = base + 32 * k;
        const bool isl = v[k] < kQ, ish = v[k] > kQ;
        const uint32_t lm = __ballot_sync(0xFFFFFFFFu, isl), hm = __ballot_sync(0xFFFFFFFFu, ish);
        if (lm) {
            const uint64_t inc = warp_incl(isl ? kQ - v[k] : 0ull, lane);
            if (isl) {
                const uint32_t r = at.a + __popc(lm & lt);
                light[r] = make_uint2((uint32_t)i, (uint32_t)v[k]);
                dp[r] = at.c + inc;
            }
            at.a += __popc(lm);
            at.c += __shfl_sync(0xFFFFFFFFu, inc, 31);
        }
        if (hm) {
            const uint64_t inc = warp_incl(ish ? v[k] - kQ : 0ull, lane);
            if (ish) {
                const uint32_t r = at.b + __popc(hm & lt);
                heavy_idx[r] = (uint32_t)i;
                ep[r] = at.d + inc;
            }
            at.b += __popc(hm);
            at.d += __shfl_sync(0xFFFFFFFFu, inc, 31);
        }
        if (!isl && !ish && i < n) tab[i] = make_uint2(kThrFull, (uint32_t)i);
    }
}

__device__ __forceinline__ uint32_t lower_bound_u64(const uint64_t* a, uint32_t n, uint64_t v) {
    uint32_t lo = 0, hi = n;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}
__device__ __forceinline__ uint32_t upper_bound_u64(const uint64_t* a, uint32_t n, uint64_t v) {
    uint32_t lo = 0, hi = n;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a[mid] <= v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// first[g]: the first heavy item that tops up light g kPairTile, or H past
// the last; one thread per group of lights.
constexpr int kPairTile = 1024;

__global__ void k_pair_starts(const Quad* total, const uint64_t* __restrict__ dp, const uint64_t* __restrict__ ep,
                              uint32_t* __restrict__ first) {
    const uint32_t L = total->a, H = total->b, groups = (L + kPairTile - 1) / kPairTile;
    for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g <= groups; g += gridDim.x * blockDim.x) {
        const uint32_t j = g * kPairTile;
        first[g] = g == groups ? H : lower_bound_u64(ep, H, j ? dp[j - 1] : 0ull);
    }
}

// The lights' buckets.  The heavies that a group of 1,024 consecutive lights
// needs are consecutive too: searched in shared memory when they fit (about
// 100 of them on R-MAT 20), instead of 22 steps through all heavies in L2 for
// every light (588 us for 31.4M arcs; 185 like this).
constexpr uint32_t kPairWindow = 2048;

__global__ void __launch_bounds__(256) k_pair_lights(const Quad* total, const uint2* __restrict__ light,
                                                     const uint64_t* __restrict__ dp, const uint32_t* __restrict__ heavy_idx,
                                                     const uint64_t* __restrict__ ep, const uint32_t* __restrict__ first,
                                                     uint2* __restrict__ tab, uint32_t* status) {
    __shared__ uint64_t win[kPairWindow];
    const uint32_t L = total->a, H = total->b, groups = (L + kPairTile - 1) / kPairTile;
    for (uint32_t g = blockIdx.x; g < groups; g += gridDim.x) {
        // the heavies k with EP[k-1] < DP of the group's lights: [k0, k1]
        const uint32_t k0 = first[g], k1 = min(first[g + 1], H ? H - 1u : 0u), nk = k1 >= k0 ? k1 - k0 + 1u : 0u;
        const bool held = nk <= kPairWindow;
        __syncthreads();
        if (held)
            for (uint32_t k = threadIdx.x; k < nk; k += blockDim.x) win[k] = ep[k0 + k];
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kPairTile / 256; ++q) {
            const uint32_t j = g * kPairTile + q * 256 + threadIdx.x;
            if (j >= L) continue;
            const uint64_t dpex = j ? dp[j - 1] : 0ull;
            const uint32_t k = k0 + (held ? lower_bound_u64(win, nk, dpex) : lower_bound_u64(ep + k0, nk, dpex));
            if (k >= H || k > k1) {
                atomicOr(status, DEV_ERR_ALIAS);
                continue;
            }
            const uint2 l = light[j];
            tab[l.x] = make_uint2(l.y, heavy_idx[k]);
        }
    }
}

__global__ void k_pair_heavies(const Quad* total, const uint64_t* __restrict__ dp, const uint32_t* __restrict__ heavy_idx,
                               const uint64_t* __restrict__ ep, uint2* __restrict__ tab, uint32_t* status) {
    const uint32_t L = total->a, H = total->b;
    for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < H; k += gridDim.x * blockDim.x) {
        const uint32_t i = heavy_idx[k];
        if (k + 1 == H) {
            // the totals of deficits and excesses must agree exactly
            if (L == 0 || dp[L - 1] != ep[k]) atomicOr(status, DEV_ERR_ALIAS);
            tab[i] = make_uint2(kThrFull, i);
            continue;
        }
        const uint32_t j = upper_bound_u64(dp, L, ep[k]);
        if (j >= L || dp[j] - ep[k] > kQ) {
            atomicOr(status, DEV_ERR_ALIAS);
            continue;
        }
        tab[i] = make_uint2((uint32_t)(kQ - (dp[j] - ep[k])), heavy_idx[k + 1]);
    }
}

inline unsigned grid_for(int64_t n, int threads, int64_t cap = 152 * 32) {
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (unsigned)b;
}

inline size_t align_up(size_t v) { return (v + 255) & ~size_t(255); }

}  // namespace

size_t fixed_sum_tmp_bytes(int64_t n) {
    size_t total = 0;
    int64_t cur = n;
    do {
        cur = (cur + kSumBlock - 1) / kSumBlock;
        total += align_up(sizeof(double) * (size_t)(cur > 0 ? cur : 1));
    } while (cur > 1);
    return total;
}

cudaError_t fixed_sum_f64(const double* x, int64_t n, double* tmp, double* out, cudaStream_t s) {
    if (n <= 0) return cudaMemsetAsync(out, 0, sizeof(double), s);
    const double* in = x;
    int64_t cur = n;
    char* p = (char*)tmp;
    while (true) {
        const int64_t nb = (cur + kSumBlock - 1) / kSumBlock;
        double* dst = nb == 1 ? out : (double*)p;
        k_tree_sum<double><<<(unsigned)((nb + 7) / 8), 256, 0, s>>>(in, cur, dst);
        if (nb == 1) break;
        p += align_up(sizeof(double) * (size_t)nb);
        in = dst;
        cur = nb;
    }
    return cudaGetLastError();
}

cudaError_t fixed_sums_f64(const double* x, int64_t rows, int64_t padded, double* tmp, double* out, cudaStream_t s) {
    const int64_t nb = padded / kSumBlock;  // (at most kSumBlock)
    if (padded % kSumBlock || nb > kSumBlock) return cudaErrorInvalidValue;
    k_tree_sum<double><<<(unsigned)((rows * nb + 7) / 8), 256, 0, s>>>(x, rows * padded, tmp);
    k_tree_rows<<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(tmp, rows, nb, out);
    return cudaGetLastError();
}

cudaError_t scan_graph(int64_t n_nodes, int64_t n_arcs, const int32_t* src, const int32_t* dst, const float* w,
                       int64_t* row_ptr, unsigned long long* degi, GraphScan* out, uint32_t* status, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(degi, 0, sizeof(unsigned long long) * (size_t)n_nodes, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(out, 0, sizeof(GraphScan), s);
    if (e != cudaSuccess) return e;
    k_graph_scan<<<grid_for((n_arcs + kArcs - 1) / kArcs, 256, 152 * 32), 256, 0, s>>>(n_nodes, n_arcs, src, dst, w, row_ptr,
                                                                                      degi, out, status);
    return cudaGetLastError();
}

cudaError_t neg_weights(int64_t n_nodes, const int64_t* row_ptr, const float* w, const unsigned long long* degi, bool whole,
                        double* x, float* deg, cudaStream_t s) {
    if (whole) k_neg_weights_int<<<grid_for(n_nodes, 256), 256, 0, s>>>(n_nodes, degi, x, deg);
    else k_neg_weights<<<grid_for(n_nodes, 128, 1 << 20), 128, 0, s>>>(n_nodes, row_ptr, w, x, deg);
    return cudaGetLastError();
}

// tmp layout: W | counters | m[n] | dp[n] | ep[n] | light[n] | heavy_idx[n] |
//             scan tiles (u32) | class tiles (Quad) | pair starts | fixed-sum tmp
size_t alias_build_tmp_bytes(int64_t n) {
    const int64_t nt = scan_tiles(n) + 1, nc = (n + kClassTile - 1) / kClassTile + 1;
    return align_up(sizeof(double)) + align_up(sizeof(MassCounters)) + 3 * align_up(sizeof(uint64_t) * n) +
           align_up(sizeof(uint2) * n) + align_up(sizeof(uint32_t) * n) + align_up(sizeof(uint32_t) * nt) +
           align_up(sizeof(Quad) * nc) + align_up(sizeof(uint32_t) * (n / kPairTile + 2)) + fixed_sum_tmp_bytes(n);
}

// x: the weights, T = double, or float (arc weights; null: all 1).  total
// (nullable, host): their fixed-order FP64 sum where it is known; whole: the
// weights are integers (T = float).
template <typename T>
static cudaError_t build(const T* x, int64_t n, const double* total_w, bool whole, uint2* tab, void* tmp, uint32_t* status,
                         cudaStream_t s) {
    char* p = (char*)tmp;
    auto take = [&](size_t bytes) {
        char* r = p;
        p += align_up(bytes);
        return (void*)r;
    };
    const int64_t nt = scan_tiles(n) + 1, nc = (n + kClassTile - 1) / kClassTile;
    double* W = (double*)take(sizeof(double));
    MassCounters* cnt = (MassCounters*)take(sizeof(MassCounters));
    uint64_t* m = (uint64_t*)take(sizeof(uint64_t) * n);
    uint64_t* dp = (uint64_t*)take(sizeof(uint64_t) * n);
    uint64_t* ep = (uint64_t*)take(sizeof(uint64_t) * n);
    uint2* light = (uint2*)take(sizeof(uint2) * n);
    uint32_t* heavy_idx = (uint32_t*)take(sizeof(uint32_t) * n);
    uint32_t* tiles32 = (uint32_t*)take(sizeof(uint32_t) * nt);
    Quad* tilesQ = (Quad*)take(sizeof(Quad) * (nc + 1));
    uint32_t* starts = (uint32_t*)take(sizeof(uint32_t) * (n / kPairTile + 2));
    double* sum_tmp = (double*)p;

    cudaError_t e;
    if (total_w) {
        if ((e = cudaMemcpyAsync(W, total_w, sizeof(double), cudaMemcpyHostToDevice, s)) != cudaSuccess) return e;
    } else if constexpr (sizeof(T) == 8) {
        if ((e = fixed_sum_f64(x, n, sum_tmp, W, s)) != cudaSuccess) return e;
    } else {
        // the first level reads the FP32 weights, the others its FP64 sums
        const int64_t nb = (n + kSumBlock - 1) / kSumBlock;
        double* dst = nb == 1 ? W : sum_tmp;
        k_tree_sum<T><<<(unsigned)((nb + 7) / 8), 256, 0, s>>>(x, n, dst);
        if (nb > 1 &&
            (e = fixed_sum_f64(dst, nb, (double*)((char*)sum_tmp + align_up(sizeof(double) * (size_t)nb)), W, s)) != cudaSuccess)
            return e;
    }
    if ((e = cudaMemsetAsync(cnt, 0, sizeof(MassCounters), s)) != cudaSuccess) return e;
    k_masses<T><<<grid_for(n, 256, 152 * 8), 256, 0, s>>>(n, x, W, whole, m, cnt, status);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    MassCounters h;
    if ((e = cudaMemcpyAsync(&h, cnt, sizeof(h), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    const uint64_t target = (uint64_t)n * kQ;
    const int64_t D = (int64_t)(target - (uint64_t)h.sum_m);
    Mass mass{m, 0, 0};
    if (D > 0) {
        if (h.npos == 0) {
            uint32_t bit = DEV_ERR_ALIAS;
            return cudaMemcpyAsync(status, &bit, sizeof(bit), cudaMemcpyHostToDevice, s);
        }
        const uint64_t q = (uint64_t)D / h.npos, r = (uint64_t)D % h.npos;
        if (h.npos == (unsigned long long)n) {
            // every weight is positive: an item's rank is its index, and the
            // remainder is added where the masses are read
            mass.q = q;
            mass.r = r;
        } else if constexpr (sizeof(T) == 8) {
            OutAddRR out{x, m, q, r};
            if ((e = device_scan<uint32_t>(n, GenPos{x}, out, tiles32, s)) != cudaSuccess) return e;
        } else {
            uint32_t bit = DEV_ERR_ALIAS;  // (arc weights are all positive)
            return cudaMemcpyAsync(status, &bit, sizeof(bit), cudaMemcpyHostToDevice, s);
        }
    } else if (D < 0) {
        if ((uint64_t)(-D) > h.nge1) {
            uint32_t bit = DEV_ERR_ALIAS;
            return cudaMemcpyAsync(status, &bit, sizeof(bit), cudaMemcpyHostToDevice, s);
        }
        OutSubFirst out{m, (uint64_t)(-D)};
        if ((e = device_scan<uint32_t>(n, GenGe1{m}, out, tiles32, s)) != cudaSuccess) return e;
    }
    k_class_sums<<<(unsigned)nc, 256, 0, s>>>(n, mass, tilesQ);
    k_scan_tiles<Quad><<<1, 1024, 0, s>>>(nc, tilesQ, tilesQ + nc);
    k_class_apply<<<(unsigned)nc, 256, 0, s>>>(n, mass, tilesQ, light, dp, heavy_idx, ep, tab);
    const Quad* total = tilesQ + nc;
    k_pair_starts<<<grid_for(n / kPairTile + 1, 128), 128, 0, s>>>(total, dp, ep, starts);
    k_pair_lights<<<grid_for((n + kPairTile - 1) / kPairTile, 1, 152 * 32), 256, 0, s>>>(total, light, dp, heavy_idx, ep,
                                                                                        starts, tab, status);
    k_pair_heavies<<<grid_for(n, 256), 256, 0, s>>>(total, dp, heavy_idx, ep, tab, status);
    return cudaGetLastError();
}

cudaError_t alias_build(const double* x, int64_t n, uint2* tab, void* tmp, uint32_t* status, cudaStream_t s) {
    return build<double>(x, n, nullptr, false, tab, tmp, status, s);
}
cudaError_t alias_build_arcs(const float* w, int64_t n, const double* total_w, bool whole, uint2* tab, void* tmp,
                             uint32_t* status, cudaStream_t s) {
    return build<float>(w, n, total_w, whole, tab, tmp, status, s);
}

}  // namespace line
