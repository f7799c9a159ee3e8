// Row access shared by the training kernels (train.cu, hogwild.cu): the
// lane geometry of a row, FP32/BF16 row loads, and row stores with BF16
// stochastic rounding.
#pragma once

#include "line_internal.cuh"

namespace line {

// ---------------------------------------------------------------------------
// Row geometry: a row of D values is handled by L lanes, E values per lane,
// moved as vectors of 4 values (16 bytes of FP32, 8 bytes of BF16).
// ---------------------------------------------------------------------------
// (host and device share these two: the work-item map of the persistent
// schedule is laid out on the host)
constexpr int geom_vec(int /*dtype*/) { return 4; }
constexpr int geom_lanes(int dim, int dtype) { return dim / geom_vec(dtype) < 32 ? dim / geom_vec(dtype) : 32; }

template <int D, int DT>
struct Geom {
    static constexpr int VEC = geom_vec(DT);
    static constexpr int L = geom_lanes(D, DT);
    static constexpr int E = D / L;
    static constexpr int NV = E / VEC;
    static constexpr int GPW = 32 / L;  // lane groups per warp
    static_assert(D % (VEC * L) == 0 && NV >= 1, "unsupported dim");
};

template <int D, int DT>
__device__ __forceinline__ void load_row(const void* table, int64_t row, int lig, float (&v)[Geom<D, DT>::E]) {
    using G = Geom<D, DT>;
    if constexpr (DT == LINE_DTYPE_F32) {
        const float4* p = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(table) + row * D + lig * G::E);
#pragma unroll
        for (int q = 0; q < G::NV; ++q) {
            const float4 a = ld_cg(p + q);
            v[4 * q] = a.x;
            v[4 * q + 1] = a.y;
            v[4 * q + 2] = a.z;
            v[4 * q + 3] = a.w;
        }
    } else {
        const uint2* p = reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(table) + row * D + lig * G::E);
#pragma unroll
        for (int q = 0; q < G::NV; ++q) {
            const uint2 a = __ldcg(p + q);
            v[4 * q] = __uint_as_float(a.x << 16);
            v[4 * q + 1] = __uint_as_float(a.x & 0xFFFF0000u);
            v[4 * q + 2] = __uint_as_float(a.y << 16);
            v[4 * q + 3] = __uint_as_float(a.y & 0xFFFF0000u);
        }
    }
}

// MurmurHash3's 32-bit finaliser (Appleby).
__device__ __forceinline__ uint32_t fmix32(uint32_t h) {
    h ^= h >> 16;
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    h *= 0xC2B2AE35u;
    h ^= h >> 16;
    return h;
}

// Random bits for the stochastic rounding of the rows written by the batch
// that starts at sample t0.  The batch's salt is the low half of the
// SplitMix64 output function (Steele, Lea, Flood, OOPSLA 2014) of
// seed ^ t0 0x9E3779B97F4A7C15; the 64 bits for the 4 values at columns
// 4 k4 .. 4 k4 + 3 of `row` of table `table_id` are the words
// w_j = fmix32(salt + (2 row + table) 0x9E3779B1 + 2 k4 + j), j = 0 (low) and
// 1 (high).
__device__ __forceinline__ uint32_t sr_salt(uint64_t seed, uint64_t t0) {
    uint64_t s = seed ^ (t0 * 0x9E3779B97F4A7C15ull);
    s = (s ^ (s >> 30)) * 0xBF58476D1CE4E5B9ull;
    s = (s ^ (s >> 27)) * 0x94D049BB133111EBull;
    return (uint32_t)(s ^ (s >> 31));
}
__device__ __forceinline__ uint2 sr_words(uint32_t salt, uint32_t table_id, uint64_t row, uint32_t k4) {
    const uint32_t base = salt + (uint32_t)(2 * row + table_id) * 0x9E3779B1u + 2u * k4;
    return make_uint2(fmix32(base), fmix32(base + 1u));
}

// Store a row part; BF16 rounds stochastically: value i of a 4-value vector
// adds bits [16 i, 16 i + 16) of sr_words(...) below the BF16 mantissa, then
// truncates (two values per cvt.rs instruction).
template <int D, int DT>
__device__ __forceinline__ void store_row(void* table, int64_t row, int lig, const float (&v)[Geom<D, DT>::E],
                                          uint32_t salt, uint32_t table_id) {
    using G = Geom<D, DT>;
    if constexpr (DT == LINE_DTYPE_F32) {
        float4* p = reinterpret_cast<float4*>(reinterpret_cast<float*>(table) + row * D + lig * G::E);
#pragma unroll
        for (int q = 0; q < G::NV; ++q) st_cg(p + q, make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
    } else {
        uint2* p = reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(table) + row * D + lig * G::E);
#pragma unroll
        for (int q = 0; q < G::NV; ++q) {
            const uint2 r = sr_words(salt, table_id, (uint64_t)row, (uint32_t)((lig * G::E + 4 * q) >> 2));
            __stcg(p + q, make_uint2(bf16x2_sr(v[4 * q], v[4 * q + 1], r.x), bf16x2_sr(v[4 * q + 2], v[4 * q + 3], r.y)));
        }
    }
}

// Packed FP32 arithmetic on E values (two per instruction on sm_100 and
// later, each half rounded as the scalar instruction would be).
// r = a b + c
template <int E>
__device__ __forceinline__ void vfma(float (&r)[E], float a, const float (&b)[E], const float (&c)[E]) {
#pragma unroll
    for (int e = 0; e < E; e += 2) {
        const float2 t = __ffma2_rn(make_float2(a, a), make_float2(b[e], b[e + 1]), make_float2(c[e], c[e + 1]));
        r[e] = t.x;
        r[e + 1] = t.y;
    }
}
// r = a b
template <int E>
__device__ __forceinline__ void vmul(float (&r)[E], float a, const float (&b)[E]) {
#pragma unroll
    for (int e = 0; e < E; e += 2) {
        const float2 t = __fmul2_rn(make_float2(a, a), make_float2(b[e], b[e + 1]));
        r[e] = t.x;
        r[e + 1] = t.y;
    }
}

// Sums of N values over the L lanes of a group, each in the order of the
// butterfly (lane distances L/2 .. 1) and so with the same bits, but each
// total only in some lanes: at every distance a lane gives away half of its
// values and receives its partner's half of the others, so N values cost
// about N + log2 L shuffles instead of N log2 L.  After reduce(), value j is
// in s[slot(j)] of lane lane(j) (and of the lanes that differ from it outside
// the distances that split it); kept() values a lane remain.
template <int L, int N>
struct Transposed {
    static constexpr int kept() {
        int n = N;
        for (int o = L / 2; o >= 1; o >>= 1) n = n > 1 ? (n + 1) / 2 : n;
        return n;
    }
    static constexpr int find(int j, bool want_lane) {
        int n = N, lane = 0;
        for (int o = L / 2; o >= 1; o >>= 1) {
            if (n <= 1) continue;
            const int half = (n + 1) / 2;
            if (j >= half) {
                lane |= o;
                j -= half;
            }
            n = half;
        }
        return want_lane ? lane : j;
    }
    static constexpr int lane(int j) { return find(j, true); }
    static constexpr int slot(int j) { return find(j, false); }
    // lanes that hold value 0 in slot 0: those with none of these bits
    static constexpr int split() {
        int n = N, m = 0;
        for (int o = L / 2; o >= 1; o >>= 1) {
            if (n > 1) m |= o;
            n = n > 1 ? (n + 1) / 2 : n;
        }
        return m;
    }
    template <typename V>
    static __device__ __forceinline__ void reduce(V (&s)[N], int lig) {
        int n = N;
#pragma unroll
        for (int o = L / 2; o >= 1; o >>= 1) {
            const bool hi = (lig & o) != 0;
            const int half = (n + 1) / 2;
#pragma unroll
            for (int i = 0; i < (N + 1) / 2; ++i) {
                if (i >= half) continue;
                if (i + half < n) {
                    const V keep = hi ? s[i + half] : s[i], give = hi ? s[i] : s[i + half];
                    s[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
                } else {
                    s[i] += __shfl_xor_sync(0xFFFFFFFFu, s[i], o);
                }
            }
            n = half;
        }
    }
};

template <int L>
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
    for (int o = L / 2; o >= 1; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

template <int L>
__device__ __forceinline__ uint32_t group_mask(int grp) {
    return L == 32 ? 0xFFFFFFFFu : (((1u << L) - 1u) << (grp * L));
}

}  // namespace line
