// Negative-sampling LINE loss over a fixed set of samples (draw domain 3):
// terms[t] = -(log sigma(s+) + sum_j log sigma(-s-_j)), s = U[u].Ctx[y] from
// the stored values, summed in 64-bit integers (FP64 where that would be less
// exact) and rounded to FP64.  The caller reduces terms[] with the
// fixed-order FP64 sum, so the loss is reproducible.
#include <math.h>

#include <algorithm>

#include "line_internal.cuh"
#include "rows.cuh"

namespace line {

namespace {

// log sigma(s) = -(max(-s, 0) + log1p(exp(-|s|)))
__device__ __forceinline__ double log_sigmoid(double s) {
    const double a = s < 0.0 ? -s : 0.0;
    return -(a + log1p(exp(-fabs(s))));
}

template <int DT>
__device__ __forceinline__ uint32_t load_bits(const void* p, int64_t idx) {
    if constexpr (DT == LINE_DTYPE_F32) return __ldg(reinterpret_cast<const uint32_t*>(p) + idx);
    else return (uint32_t)__ldg(reinterpret_cast<const unsigned short*>(p) + idx) << 16;
}

// FP32 bits of N consecutive values, idx a multiple of N.
template <int N, int DT>
__device__ __forceinline__ void load_bits(const void* p, int64_t idx, uint32_t (&b)[N]) {
    if constexpr (N == 1) {
        b[0] = load_bits<DT>(p, idx);
    } else {
        constexpr int W = DT == LINE_DTYPE_F32 ? N : N / 2;  // 32-bit words
        uint32_t w[W];
        const uint32_t* q = reinterpret_cast<const uint32_t*>(p) + (DT == LINE_DTYPE_F32 ? idx : idx / 2);
        if constexpr (W == 1) {
            w[0] = __ldg(q);
        } else if constexpr (W == 2) {
            const uint2 v = __ldg(reinterpret_cast<const uint2*>(q));
            w[0] = v.x;
            w[1] = v.y;
        } else {
#pragma unroll
            for (int k = 0; k < W; k += 4) {
                const uint4 v = __ldg(reinterpret_cast<const uint4*>(q) + k / 4);
                w[k] = v.x;
                w[k + 1] = v.y;
                w[k + 2] = v.z;
                w[k + 3] = v.w;
            }
        }
#pragma unroll
        for (int k = 0; k < N; ++k) b[k] = DT == LINE_DTYPE_F32 ? w[k * W / N] : (k & 1) ? w[k / 2] & 0xFFFF0000u : w[k / 2] << 16;
    }
}

// A dot of FP32 rows in integers, IT products a lane: the 48-bit products of
// the significands, SH bits above their last one, each shifted down by its
// exponent's distance to the largest exponent's, to nearest, and summed
// exactly.  A product is off by at most half a unit of 2^-(46 + SH) of the one
// with the largest exponent, the dot by half of D units: 2^-56, 2^-55, 2^-54,
// 2^-52 and 2^-51 of it for D = 16, 32, 64, 128 and 256.  Against the exact
// dot over rows of normal, positive, widely spread and trained values and of
// one product above all others, 2^9 to 2^62 times, the rms and the largest
// error are below the FP64 chain's at every width, by 2 to 20 times at D >= 64
// for rows whose sum cancels, by 1 to 4 times for the others.  (Rounded down,
// the small products beside one large one all counted on one side: 2^-52 of it
// at D = 128, where the chain was exact.)  A subnormal factor has no leading
// bit, and its product would be held to fewer: such rows take FP64 sums.
template <int IT>
struct Fixed {
    // a lane's sum (of twice the products up to IT = 4) stays below 2^63, each
    // factor below 2^31
    static constexpr int SH = IT <= 2 ? 13 : 12;
    static constexpr int CUT = 27;       // limbs of the sum over 32 lanes: 32 2^27 fits 32 bits

    // This lane's part of a dot; `top`: the largest product's exponent (of all
    // lanes; twice biased, in place); `wide`: |= an infinity, a NaN or a
    // subnormal value was met.
    static __device__ __forceinline__ int64_t lane_sum(const uint32_t (&a)[IT], const uint32_t (&b)[IT], uint32_t& top, bool& wide) {
        int64_t p[IT];
        uint32_t ex[IT], m = 0, mx = 0, mn = 0xFFFFFFFFu;
#pragma unroll
        for (int k = 0; k < IT; ++k) {
            const uint32_t ea = a[k] & 0x7F800000u, eb = b[k] & 0x7F800000u;
            mx = max(mx, max(ea, eb));
            // (0 for a zero, below 2^23 for a subnormal)
            const uint32_t sa = (a[k] & 0x7FFFFFu) | min(ea, 0x800000u), sb = (b[k] & 0x7FFFFFu) | min(eb, 0x800000u);
            mn = min(mn, min(sa - 1u, sb - 1u));
            constexpr int UP = SH - 7 + (IT <= 4);
            const int32_t sg = (int32_t)(a[k] ^ b[k]) < 0 ? -(1 << UP) : 1 << UP;
            p[k] = (int64_t)(int32_t)(sa << 7) * ((int32_t)sb * sg);
            ex[k] = p[k] ? ea + eb : 0u;
            m = max(m, ex[k]);
        }
        wide |= mx >= 0x7F800000u || mn < 0x7FFFFFu;
        top = __reduce_max_sync(0xFFFFFFFFu, m);
        int64_t sum = 0;
#pragma unroll
        for (int k = 0; k < IT; ++k) {
            const uint32_t s = min((top - ex[k]) >> 23, 63u);
            if constexpr (IT <= 4) {
                // twice the product, rounded down: t; to nearest it is (t + (t & 1)) / 2
                const int64_t t = p[k] >> s;
                sum += t + (t & 1);
            } else {
                sum += (p[k] + (int64_t)((uint64_t)1 << s >> 1)) >> s;
            }
        }
        return IT <= 4 ? sum >> 1 : sum;
    }
    // The dot from the limbs' sums over the lanes.
    static __device__ __forceinline__ double value(int64_t h, uint32_t lo, uint32_t top) {
        const int e = (int)(top >> 23) - 300 - SH;
        return fma((double)h, (double)(1u << CUT), (double)lo) * __hiloint2double((1023 + e) << 20, 0);
    }
};

// One warp for a group of samples whose K+1 scores each fill its lanes (one
// sample where K+1 > 32, in rounds of 32 scores).  Lane q draws its score's
// row; the dots are taken N at a time with all lanes on one, IT consecutive
// values a lane, in integers (Fixed); their limbs are reduced by transposed
// butterflies (each total in some lanes only); then every lane evaluates the
// log-sigmoid of its own score, and a sample's are subtracted in order.  Rows
// with infinities, NaNs or subnormals take FP64 sums, value k of a row in lane
// k mod 32.
// Bound: issue slots of the integer dots (about 33 instructions a product) and
// GB300's FP64 pipe in the log-sigmoids (two lanes a clock and SM, also for
// conversions).  N = 3 at 64 registers keeps four blocks resident (8 at 117
// registers: 1.85 ms, 4: 1.48).
// One warp per sample, with all lanes on the same log-sigmoid and FP64
// conversions of every value, took 25.2 ms for 2^20 samples of K = 5, d = 128
// FP32; FP64 sums of values widened by integer instructions 2.77; this 1.52
// (1.40 without the rounding and the look for subnormals).
template <int D, int DT>
__global__ void __launch_bounds__(256, 4) k_loss_terms(const void* __restrict__ U, const void* __restrict__ Ctx, int K,
                                                    const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                    const uint2* __restrict__ edge_tab, int64_t n_arcs,
                                                    const uint2* __restrict__ neg_tab, int64_t n_nodes, uint64_t seed,
                                                    int64_t m, double* __restrict__ terms) {
    constexpr int IT = D >= 32 ? D / 32 : 1;
    constexpr int N = D > 128 ? 2 : 3;
    using F = Fixed<IT>;
    const int lane = threadIdx.x & 31;
    const bool holds = lane < D;
    const int C1 = K + 1, S = C1 <= 32 ? 32 / C1 : 1;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t t0 = S * (blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5)); t0 < m; t0 += S * warps) {
        const int live = (int)min((int64_t)S, m - t0);
        double L = 0.0;
        int64_t u0 = 0;  // the sample's source (more than one round: from the first)
        for (int j0 = 0; j0 < C1; j0 += 32) {
            const int nq = C1 <= 32 ? live * C1 : min(32, C1 - j0);
            int64_t u = u0, y = 0;
            const int smp = C1 <= 32 ? lane / C1 : 0, j = C1 <= 32 ? lane - smp * C1 : j0 + lane;
            if (lane < nq) {
                const uint4 w = draw_words(seed, 3u, (uint64_t)(t0 + smp), (uint32_t)j);
                if (j == 0) {
                    const uint32_t e = alias_pick(edge_tab, (uint64_t)n_arcs, w);
                    u = src[e];
                    y = dst[e];
                } else {
                    y = alias_pick(neg_tab, (uint64_t)n_nodes, w);
                }
            }
            if (j0 == 0) {
                u = __shfl_sync(0xFFFFFFFFu, u, lane < nq ? lane - j : 0);
                u0 = u;  // (C1 > 32: the same in every lane)
            }
            int64_t h = 0;
            uint32_t lo = 0, top = 0;
            bool direct = false;  // h holds the score's bits
            for (int q0 = 0; q0 < nq; q0 += N) {
                int64_t part[N];
                uint32_t low[N], tops[N];
                uint32_t a[N][IT], c[N][IT];
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const int q = min(q0 + i, nq - 1);
                    const int64_t uq = __shfl_sync(0xFFFFFFFFu, u, q), yq = __shfl_sync(0xFFFFFFFFu, y, q);
                    if (holds) {
                        load_bits<IT, DT>(U, uq * D + lane * IT, a[i]);
                        load_bits<IT, DT>(Ctx, yq * D + lane * IT, c[i]);
                    } else {
#pragma unroll
                        for (int k = 0; k < IT; ++k) a[i][k] = c[i][k] = 0u;
                    }
                }
                bool wide = false;
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const int64_t sum = F::lane_sum(a[i], c[i], tops[i], wide);
                    low[i] = (uint32_t)sum & ((1u << F::CUT) - 1u);
                    part[i] = sum >> F::CUT;
                }
                if (__any_sync(0xFFFFFFFFu, wide)) {
#pragma unroll 1
                    for (int i = 0; i < N; ++i) {
                        const int q = min(q0 + i, nq - 1);
                        const int64_t uq = __shfl_sync(0xFFFFFFFFu, u, q), yq = __shfl_sync(0xFFFFFFFFu, y, q);
                        double v = 0.0;
                        for (int k = 0; k < IT; ++k) {
                            const uint32_t x = holds ? load_bits<DT>(U, uq * D + k * 32 + lane) : 0u;
                            const uint32_t z = holds ? load_bits<DT>(Ctx, yq * D + k * 32 + lane) : 0u;
                            v = fma((double)__uint_as_float(x), (double)__uint_as_float(z), v);
                        }
#pragma unroll
                        for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
                        if (lane == q0 + i) {
                            h = __double_as_longlong(v);
                            direct = true;
                        }
                    }
                    continue;
                }
                using T = Transposed<32, N>;
                T::reduce(part, lane);
                T::reduce(low, lane);
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const int64_t vh = __shfl_sync(0xFFFFFFFFu, part[0], T::lane(i));
                    const uint32_t vl = __shfl_sync(0xFFFFFFFFu, low[0], T::lane(i));
                    if (lane == q0 + i) {
                        h = vh;
                        lo = vl;
                        top = tops[i];
                    }
                }
            }
            const double score = direct ? __longlong_as_double(h) : F::value(h, lo, top);
            const double ls = lane < nq ? log_sigmoid(j == 0 ? score : -score) : 0.0;
            const int per = C1 <= 32 ? C1 : nq;
            for (int k = 0; k < per; ++k) L -= __shfl_sync(0xFFFFFFFFu, ls, min(lane * C1, 31) + k & 31);
        }
        if (lane < live) terms[t0 + lane] = L;
    }
}

template <int D>
cudaError_t launch_terms(int dtype, unsigned blocks, const void* U, const void* Ctx, int K, const int32_t* src,
                         const int32_t* dst, const uint2* edge_tab, int64_t n_arcs, const uint2* neg_tab, int64_t n_nodes,
                         uint64_t seed, int64_t m, double* terms, cudaStream_t s) {
    if (dtype == LINE_DTYPE_F32)
        k_loss_terms<D, LINE_DTYPE_F32><<<blocks, 256, 0, s>>>(U, Ctx, K, src, dst, edge_tab, n_arcs, neg_tab, n_nodes,
                                                               seed, m, terms);
    else
        k_loss_terms<D, LINE_DTYPE_BF16><<<blocks, 256, 0, s>>>(U, Ctx, K, src, dst, edge_tab, n_arcs, neg_tab, n_nodes,
                                                                seed, m, terms);
    return cudaGetLastError();
}

}  // namespace

cudaError_t eval_loss_terms(const void* U, const void* Ctx, int dtype, int dim, int K, const int32_t* src,
                            const int32_t* dst, const uint2* edge_tab, int64_t n_arcs, const uint2* neg_tab,
                            int64_t n_nodes, uint64_t seed, int64_t m, double* terms, cudaStream_t s) {
    if (m <= 0) return cudaSuccess;
    const int64_t S = K + 1 <= 32 ? 32 / (K + 1) : 1;  // samples a warp takes at once
    const unsigned blocks = (unsigned)std::min<int64_t>((m + 8 * S - 1) / (8 * S), 152 * 32);
    switch (dim) {
        case 16: return launch_terms<16>(dtype, blocks, U, Ctx, K, src, dst, edge_tab, n_arcs, neg_tab, n_nodes, seed, m, terms, s);
        case 32: return launch_terms<32>(dtype, blocks, U, Ctx, K, src, dst, edge_tab, n_arcs, neg_tab, n_nodes, seed, m, terms, s);
        case 64: return launch_terms<64>(dtype, blocks, U, Ctx, K, src, dst, edge_tab, n_arcs, neg_tab, n_nodes, seed, m, terms, s);
        case 128: return launch_terms<128>(dtype, blocks, U, Ctx, K, src, dst, edge_tab, n_arcs, neg_tab, n_nodes, seed, m, terms, s);
        case 256: return launch_terms<256>(dtype, blocks, U, Ctx, K, src, dst, edge_tab, n_arcs, neg_tab, n_nodes, seed, m, terms, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace line
