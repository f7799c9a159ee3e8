// Link-prediction evaluation (reporting): scores of node pairs and the exact
// Mann-Whitney AUC of positive against negative pairs: held-out edges
// against non-edges, the measure of embedding quality this library reports
// (the paper's own, node classification by Micro/Macro-F1 in §V-C, needs
// node labels).  Over the requested
// orders o, with z(x) = [U_o[x]]_o the concatenated rows:
//
//   dot:     score(u, v) = z(u).z(v) = sum_o U_o[u].U_o[v]
//   cosine:  score(u, v) = n(u).n(v) / (|n(u)| |n(v)|),  n(x) = [U_o[x] / |U_o[x]|]_o
//
// (cosine: an all-zero row contributes a zero block, a zero concatenated
// vector scores 0).  Scores are FP32: per order the dot and the two squared
// norms are FP32 FMA chains over a lane's dimensions, reduced by a butterfly
// (every lane ends with the same bits).  The AUC then
// counts, in integers, the (positive, negative) pairs with neg < pos and with
// neg == pos: the negatives' order-preserving 32-bit keys are radix sorted and
// every positive key is located by binary search.
#include "line_internal.cuh"
#include "rows.cuh"

namespace line {

namespace {

__device__ __forceinline__ float load_f(const void* p, int dtype, int64_t idx) {
    return dtype == LINE_DTYPE_F32 ? reinterpret_cast<const float*>(p)[idx]
                                   : __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[idx]);
}

// Monotone map float -> uint32 (after -0 -> +0): a < b  <=>  key(a) < key(b).
__device__ __forceinline__ uint32_t order_key(float f) {
    uint32_t b = __float_as_uint(f == 0.0f ? 0.0f : f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// One warp for kPairs pairs at once (their rows are in flight together);
// value k of a row in lane k mod 32, the totals by transposed butterflies:
// pair i's in lane T::lane(i) and those that differ from it in lower bits.
// D, DT: the tables' row width and type, or D = 0 where two orders' differ.
// A random-row gather (2 rows a pair and order): 3.1M pairs of two orders at
// d = 128 took 1.36 ms one pair at a time with the norms always taken, 2.24
// four at a time with the width and type read at run time (106 registers),
// 0.75 like this (6.4 GB of rows).
constexpr int kPairs = 2;

template <int SCORE, int D, int DT>
__global__ void __launch_bounds__(256) k_pair_scores(ScoreTables t, const int32_t* __restrict__ src,
                                                     const int32_t* __restrict__ dst, int64_t n, int64_t n_nodes,
                                                     float* __restrict__ scores, uint32_t* __restrict__ keys,
                                                     uint32_t* status) {
    using T = Transposed<32, kPairs>;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t i0 = kPairs * (blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5)); i0 < n; i0 += kPairs * warps) {
        int64_t u[kPairs], v[kPairs];
        bool bad[kPairs];
#pragma unroll
        for (int i = 0; i < kPairs; ++i) {
            u[i] = i0 + i < n ? src[i0 + i] : 0;
            v[i] = i0 + i < n ? dst[i0 + i] : 0;
            bad[i] = u[i] < 0 || u[i] >= n_nodes || v[i] < 0 || v[i] >= n_nodes;
            if (bad[i]) u[i] = v[i] = 0;
        }
        float zz = 0.0f, cu = 0.0f, cv = 0.0f, dd = 0.0f;
#pragma unroll
        for (int o = 0; o < 2; ++o) {
            if (o >= t.n) break;
            const void* U = t.U[o];
            const int dim = D ? D : t.dim[o], dt = D ? DT : t.dtype[o];
            float dot[kPairs], nu[kPairs], nv[kPairs];
#pragma unroll
            for (int i = 0; i < kPairs; ++i) dot[i] = nu[i] = nv[i] = 0.0f;
            auto add = [&](int k) {
#pragma unroll
                for (int i = 0; i < kPairs; ++i) {
                    const float a = load_f(U, dt, u[i] * dim + k), b = load_f(U, dt, v[i] * dim + k);
                    dot[i] = fmaf(a, b, dot[i]);
                    if (SCORE == LINE_SCORE_COSINE) {
                        nu[i] = fmaf(a, a, nu[i]);
                        nv[i] = fmaf(b, b, nv[i]);
                    }
                }
            };
            if constexpr (D >= 32) {
#pragma unroll
                for (int k = 0; k < D; k += 32) add(k + lane);
            } else {
                for (int k = lane; k < dim; k += 32) add(k);
            }
            T::reduce(dot, lane);
            dd += dot[0];
            if (SCORE == LINE_SCORE_COSINE) {
                T::reduce(nu, lane);
                T::reduce(nv, lane);
                if (nu[0] > 0.0f && nv[0] > 0.0f) zz += dot[0] / (sqrtf(nu[0]) * sqrtf(nv[0]));
                if (nu[0] > 0.0f) cu += 1.0f;
                if (nv[0] > 0.0f) cv += 1.0f;
            }
        }
        float sc = SCORE == LINE_SCORE_DOT ? dd : (cu > 0.0f && cv > 0.0f) ? zz / sqrtf(cu * cv) : 0.0f;
#pragma unroll
        for (int i = 0; i < kPairs; ++i) {
            if (lane != T::lane(i) || i0 + i >= n) continue;
            if (bad[i]) {
                atomicOr(status, DEV_ERR_INDEX);
                sc = 0.0f;
            }
            if (!(sc == sc)) atomicOr(status, DEV_ERR_VALUE);
            scores[i0 + i] = sc;
            keys[i0 + i] = order_key(sc);
        }
    }
}

using ScoreFn = void (*)(ScoreTables, const int32_t*, const int32_t*, int64_t, int64_t, float*, uint32_t*, uint32_t*);

template <int SCORE, int DT>
ScoreFn score_kernel(int dim) {
    switch (dim) {
        case 32: return k_pair_scores<SCORE, 32, DT>;
        case 64: return k_pair_scores<SCORE, 64, DT>;
        case 128: return k_pair_scores<SCORE, 128, DT>;
        case 256: return k_pair_scores<SCORE, 256, DT>;
        default: return k_pair_scores<SCORE, 0, DT>;
    }
}

template <int SCORE>
ScoreFn score_kernel(const ScoreTables& t) {
    const bool same = t.n == 1 || (t.dim[0] == t.dim[1] && t.dtype[0] == t.dtype[1]);
    const int dim = same ? t.dim[0] : 0;
    return t.dtype[0] == LINE_DTYPE_F32 ? score_kernel<SCORE, LINE_DTYPE_F32>(dim) : score_kernel<SCORE, LINE_DTYPE_BF16>(dim);
}

// ---- LSD radix sort of 32-bit keys, 8 bits per pass.  Tiles of kTile keys,
// one block each; per-tile digit counts are scanned digit-major, and the
// scatter ranks keys stably (in index order) within each tile.
constexpr int kThreads = 256;
constexpr int kRounds = 16;
constexpr int kTile = kThreads * kRounds;

__global__ void k_radix_hist(const uint32_t* __restrict__ keys, int64_t n, int shift, uint32_t* __restrict__ hist) {
    __shared__ uint32_t cnt[256];
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kTile;
    for (int r = 0; r < kRounds; ++r) {
        const int64_t i = base + r * kThreads + threadIdx.x;
        if (i < n) atomicAdd(&cnt[(keys[i] >> shift) & 0xFFu], 1u);
    }
    __syncthreads();
    hist[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = cnt[threadIdx.x];
}

// Block d: exclusive scan in place of digit d's counts over the tiles
// (hist[d tiles ..]); its total goes to tot[d].  (One block over all 256 rows
// took 189 us a pass for 1.57M keys, more than the rest of the sort.)
__global__ void __launch_bounds__(256) k_digit_scan(uint32_t* hist, int64_t n_tiles, uint32_t* __restrict__ tot) {
    __shared__ uint32_t wsum[8];
    uint32_t* row = hist + blockIdx.x * n_tiles;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t carry = 0;
    for (int64_t i0 = 0; i0 < n_tiles; i0 += 256) {
        const int64_t i = i0 + threadIdx.x;
        const uint32_t c = i < n_tiles ? row[i] : 0u;
        uint32_t x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        uint32_t before = carry, all = 0;
        for (int w = 0; w < 8; ++w) {
            if (w < warp) before += wsum[w];
            all += wsum[w];
        }
        if (i < n_tiles) row[i] = before + x - c;
        carry += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) tot[blockIdx.x] = carry;
}

__global__ void k_radix_scatter(const uint32_t* __restrict__ in, uint32_t* __restrict__ out, int64_t n, int shift,
                                const uint32_t* __restrict__ offs, const uint32_t* __restrict__ tot) {
    __shared__ uint32_t wcnt[kThreads / 32][256];
    __shared__ uint32_t run[256], wsum[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    {
        // where each digit's keys begin: the digits before it
        uint32_t x = tot[threadIdx.x];
        const uint32_t own = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        for (int w = 0; w < warp; ++w) x += wsum[w];
        run[threadIdx.x] = x - own + offs[(size_t)threadIdx.x * gridDim.x + blockIdx.x];
    }
    const int64_t base = (int64_t)blockIdx.x * kTile;
    for (int r = 0; r < kRounds; ++r) {
        for (int w = 0; w < kThreads / 32; ++w) wcnt[w][threadIdx.x] = 0;
        __syncthreads();
        const int64_t i = base + r * kThreads + threadIdx.x;
        const bool valid = i < n;
        const uint32_t key = valid ? in[i] : 0u;
        const uint32_t d = valid ? (key >> shift) & 0xFFu : 0x100u + lane;  // invalid lanes match nobody
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
        const uint32_t rank = __popc(peers & ((1u << lane) - 1u));
        if (valid && lane == 31 - __clz(peers)) wcnt[warp][d] = __popc(peers);
        __syncthreads();
        {
            // thread t owns digit t: warp offsets within the round, then the
            // digit's running position
            uint32_t s = run[threadIdx.x];
            for (int w = 0; w < kThreads / 32; ++w) {
                const uint32_t c = wcnt[w][threadIdx.x];
                wcnt[w][threadIdx.x] = s;
                s += c;
            }
            run[threadIdx.x] = s;
        }
        __syncthreads();
        if (valid) out[wcnt[warp][d] + rank] = key;
        __syncthreads();
    }
}

// counts[0] += #(neg < pos), counts[1] += #(neg == pos) over the positives.
__global__ void k_auc_count(const uint32_t* __restrict__ pos, int64_t n_pos, const uint32_t* __restrict__ neg,
                            int64_t n_neg, unsigned long long* counts) {
    unsigned long long less = 0, eq = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_pos; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t k = pos[i];
        int64_t lo = 0, hi = n_neg;
        while (lo < hi) {  // first negative >= k
            const int64_t mid = (lo + hi) >> 1;
            if (neg[mid] < k) lo = mid + 1;
            else hi = mid;
        }
        int64_t lo2 = lo, hi2 = n_neg;
        while (lo2 < hi2) {  // first negative > k
            const int64_t mid = (lo2 + hi2) >> 1;
            if (neg[mid] <= k) lo2 = mid + 1;
            else hi2 = mid;
        }
        less += (unsigned long long)lo;
        eq += (unsigned long long)(lo2 - lo);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        less += __shfl_xor_sync(0xFFFFFFFFu, less, o);
        eq += __shfl_xor_sync(0xFFFFFFFFu, eq, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(counts, less);
        atomicAdd(counts + 1, eq);
    }
}

int64_t tiles(int64_t n) { return (n + kTile - 1) / kTile; }

}  // namespace

// tmp layout: the two counters (first 256 bytes), keys [n], sort buffer
// [n_neg], digit counts [256 * tiles], digit totals [256].
size_t auc_tmp_bytes(int64_t n_pos, int64_t n_neg) {
    const int64_t n = n_pos + n_neg;
    return 256 + sizeof(uint32_t) * (size_t)(n + n_neg + 256 * (tiles(n_neg) + 1));
}

cudaError_t eval_auc(const ScoreTables& t, int score, const int32_t* src, const int32_t* dst, int64_t n_pos, int64_t n_neg,
                     int64_t n_nodes, float* scores, void* tmp, uint32_t* status, cudaStream_t s) {
    const int64_t n = n_pos + n_neg;
    unsigned long long* counts_dev = reinterpret_cast<unsigned long long*>(tmp);
    uint32_t* keys = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(tmp) + 256);
    uint32_t* alt = keys + n;
    uint32_t* hist = alt + n_neg;
    uint32_t* tot = hist + 256 * tiles(n_neg);
    cudaError_t e;
    if ((e = cudaMemsetAsync(counts_dev, 0, 2 * sizeof(unsigned long long), s)) != cudaSuccess) return e;
    {
        int64_t blocks = (n + 8 * kPairs - 1) / (8 * kPairs);
        if (blocks > 152 * 32) blocks = 152 * 32;
        const ScoreFn fn = score == LINE_SCORE_DOT ? score_kernel<LINE_SCORE_DOT>(t) : score_kernel<LINE_SCORE_COSINE>(t);
        fn<<<(unsigned)blocks, 256, 0, s>>>(t, src, dst, n, n_nodes, scores, keys, status);
    }
    // sort the negatives' keys (keys[n_pos ..]); four passes leave them in place
    uint32_t* a = keys + n_pos;
    uint32_t* b = alt;
    const int64_t nt = tiles(n_neg);
    for (int shift = 0; shift < 32; shift += 8) {
        k_radix_hist<<<(unsigned)nt, kThreads, 0, s>>>(a, n_neg, shift, hist);
        k_digit_scan<<<256, 256, 0, s>>>(hist, nt, tot);
        k_radix_scatter<<<(unsigned)nt, kThreads, 0, s>>>(a, b, n_neg, shift, hist, tot);
        uint32_t* x = a;
        a = b;
        b = x;
    }
    {
        int64_t blocks = (n_pos + 255) / 256;
        if (blocks > 152 * 8) blocks = 152 * 8;
        k_auc_count<<<(unsigned)blocks, 256, 0, s>>>(keys, n_pos, a, n_neg, counts_dev);
    }
    return cudaGetLastError();
}

}  // namespace line
