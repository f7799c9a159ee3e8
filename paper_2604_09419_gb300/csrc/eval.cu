// Negative-sampling LINE loss over a fixed set of samples (draw domain 3):
// terms[t] = -(log sigma(s+) + sum_j log sigma(-s-_j)), s = U[u].Ctx[y] in
// FP64 from the stored values.  The caller reduces terms[] with the
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

// The FP32 value with bits b as FP64, in integer instructions; `odd` is set
// for subnormals, infinities and NaNs, whose result is not valid.
__device__ __forceinline__ double widen(uint32_t b, bool& odd) {
    const uint32_t m = b & 0x7FFFFFFFu;
    odd |= m != 0u && (m < 0x00800000u || m >= 0x7F800000u);
    const uint32_t hi = (b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u);
    return __hiloint2double((int)hi, (int)(b << 29));
}

// One warp for a group of samples whose K+1 scores each fill its lanes (one
// sample where K+1 > 32, in rounds of 32 scores).  Lane q draws its score's
// row; the dots are taken eight at a time with all lanes on one, in FP64:
// value k of a row in lane k mod 32, products added in order, lanes by
// butterfly distances 16 .. 1 (transposed: each total in some lanes only);
// then every lane evaluates the log-sigmoid of its own score, and a sample's
// are subtracted in order.
// Bound: GB300's FP64 pipe (two lanes a clock and SM, also for conversions).
// One warp per sample, with all lanes on the same log-sigmoid and FP64
// conversions of every value, took 25.2 ms for 2^20 samples of K = 5, d = 128;
// this 2.77 ms.
template <int D, int DT>
__global__ void __launch_bounds__(256) k_loss_terms(const void* __restrict__ U, const void* __restrict__ Ctx, int K,
                                                    const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                    const uint2* __restrict__ edge_tab, int64_t n_arcs,
                                                    const uint2* __restrict__ neg_tab, int64_t n_nodes, uint64_t seed,
                                                    int64_t m, double* __restrict__ terms) {
    constexpr int IT = D >= 32 ? D / 32 : 1;
    constexpr int N = 8;
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
            double score = 0.0;
            for (int q0 = 0; q0 < nq; q0 += N) {
                double part[N];
                bool odd = false;
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const int q = min(q0 + i, nq - 1);
                    const int64_t uq = __shfl_sync(0xFFFFFFFFu, u, q), yq = __shfl_sync(0xFFFFFFFFu, y, q);
                    part[i] = 0.0;
#pragma unroll
                    for (int k = 0; k < IT; ++k) {
                        const uint32_t a = holds ? load_bits<DT>(U, uq * D + k * 32 + lane) : 0u;
                        const uint32_t c = holds ? load_bits<DT>(Ctx, yq * D + k * 32 + lane) : 0u;
                        part[i] = fma(widen(a, odd), widen(c, odd), part[i]);
                    }
                }
                if (__any_sync(0xFFFFFFFFu, odd)) {  // the same with the conversion instruction
#pragma unroll 1
                    for (int i = 0; i < N; ++i) {
                        const int q = min(q0 + i, nq - 1);
                        const int64_t uq = __shfl_sync(0xFFFFFFFFu, u, q), yq = __shfl_sync(0xFFFFFFFFu, y, q);
                        double v = 0.0;
                        for (int k = 0; k < IT; ++k) {
                            const uint32_t a = holds ? load_bits<DT>(U, uq * D + k * 32 + lane) : 0u;
                            const uint32_t c = holds ? load_bits<DT>(Ctx, yq * D + k * 32 + lane) : 0u;
                            v = fma((double)__uint_as_float(a), (double)__uint_as_float(c), v);
                        }
#pragma unroll
                        for (int k = 0; k < N; ++k)
                            if (k == i) part[k] = v;
                    }
                }
                using T = Transposed<32, N>;
                T::reduce(part, lane);
#pragma unroll
                for (int i = 0; i < N; ++i) {
                    const double v = __shfl_sync(0xFFFFFFFFu, part[0], T::lane(i));
                    if (lane == q0 + i) score = v;
                }
            }
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
