// Minibatch-synchronous LINE training on the GPU (Algorithm 1, Eq. 2-4).
//
// A call processes its samples in chunks of whole batches.  Per chunk:
//
//   pre-pass (index work only; it does not read the tables), on its own
//   low-priority stream so that it overlaps the previous chunk's data phase:
//     1. draws: for every sample its arc (u, v) and K negatives, kept as a
//        record (u, v, n_1..n_K): one entry, or item, per row the sample
//        touches.  Slot 0 is U[u]; slots 1..K+1 are the context rows Ctx[v],
//        Ctx[n_j] (Ctx = C for second order, U for first order; C rows get
//        ids offset by n).
//     2. per batch, the grouping of its items by row (k_group_parts; for
//        batches beyond its range a bucketing through global memory and a
//        sort per bucket): a segment is the items of one row, in (sample,
//        slot) order.  A segment with one entry is a singleton: its row is
//        read and written by one sample only.  Every (sample, slot) learns
//        its position and its segment; segments with two or more entries
//        ("shared") are listed per batch, by length class, with their first
//        position, length, row and pair count.
//
//   data phase, batch after batch:
//     gather  one lane group per sample loads U_b[u] and the K+1 context
//             rows (staged in shared memory), forms s_j = U_b[u].Ctx_b[y_j],
//             g_j = eta_b (1 - sigma(s_j)) for the positive and
//             -eta_b alpha_neg sigma(s_j) for the negatives (Algorithm 1).
//             Its contributions are slot 0: sum_j g_j Ctx_b[y_j] for U[u],
//             slot 1+j: g_j U_b[u] for Ctx[y_j].  A singleton row is written
//             back at once (Eq. 2-3); a shared row's contribution goes to the
//             delta slab at its position, so a segment's entries are
//             contiguous.  Positions count from the batch's first item: every
//             batch reuses one slab region, whose lines stay in L2 instead of
//             being written back to DRAM.
//     apply   per shared segment: the entries summed in a fixed chunked
//             order, X <- X_b - cnt eta_b lambda X_b + sum, cnt the number of
//             pair occurrences of the row (the batch-summed update of Eq. 4).
//   BF16 tables are written back with stochastic rounding (random bits from
//   a counter hash of seed, table, row, batch and column group).
//
// The order of every floating-point sum is fixed, so results are bitwise
// reproducible.  A singleton U row gets exactly the value the apply step would
// give it; a singleton context row is rounded once less, as its contribution
// g_j U_b[u] is added by a fused multiply-add.  Two schedules run the same per-sample and per-segment code:
//   LINE_MODE_BATCHED     two launches per batch, chained with programmatic
//                         dependent launch;
//   LINE_MODE_PERSISTENT  one cooperative launch per chunk: resident CTAs
//                         loop over the chunk's batches, rows staged in
//                         shared memory by bulk copies, a grid-wide barrier
//                         after each batch's gather and after its apply.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>
#include <vector>

#include "bulk.cuh"
#include "line_internal.cuh"
#include "pdl.cuh"
#include "rows.cuh"

namespace line {

// A shared segment's entries are summed in chunks of kChunk: partial sums in
// entry order, then the partials in chunk order.  Segments are listed by the
// number of their chunks: class 0 has one, classes 1, 2 and 3 up to 2, 4 and
// 8, class 4 more (the hub rows).
constexpr uint32_t kChunk = 8;
constexpr int kClasses = 5;
constexpr int kLong = kClasses;  // one more list: all of classes 1 .. 4, as they come
constexpr int kCounts = 8;       // counters of a batch: one per list, padded

__host__ __device__ inline int seg_class(uint32_t len) {
    const uint32_t c = (len + kChunk - 1) / kChunk;
    return c <= 1 ? 0 : c <= 2 ? 1 : c <= 4 ? 2 : c <= 8 ? 3 : 4;
}

// Where a batch's classes begin in its list, for at most n entries a batch.
struct SegLayout {
    uint32_t off[kClasses + 1];
    uint32_t cap;
    __host__ void set(int64_t n) {
        const uint32_t least[kClasses + 1] = {2, kChunk + 1, 2 * kChunk + 1, 4 * kChunk + 1, 8 * kChunk + 1, kChunk + 1};
        cap = 0;
        for (int c = 0; c <= kClasses; ++c) {
            off[c] = cap;
            cap += (uint32_t)(n / least[c]) + 1;
        }
    }
};

// Sort item value: (sample within the chunk) << kSlotBits | slot.
constexpr uint32_t kSlotBits = 6;
constexpr uint32_t kSlotMask = (1u << kSlotBits) - 1u;
// slot_info: a shared row's position within the batch, or kSingleBit for a row
// that the batch touches once.
constexpr uint32_t kSingleBit = 1u << 31;

// Fibonacci hashing: spreads the hot (low) row ids of skewed graphs.  The
// multiplier is odd, so hrow is a bijection of 32-bit words (inverse
// 0x0E8B2F51); within a batch items are ordered by (hrow(row), index), which
// puts them bucket by bucket (bucket = top 8 bits) and each row's entries
// together in index order.
__device__ __forceinline__ uint32_t hrow(uint32_t row) { return row * 0x9E3779B1u; }
__device__ __forceinline__ uint32_t unhrow(uint32_t h) { return h * 0x0E8B2F51u; }
__device__ __forceinline__ uint32_t bucket_of(uint32_t row) { return hrow(row) >> 24; }

// Rows a batch touches, as a bitmap of 2^kDepLog bits indexed by the top bits
// of hrow(row id) (row ids: U rows 0..n-1, C rows n..2n-1 in second order).
// A row whose bit is clear in batch b's map is not written by batch b, so it
// may be read for batch b+1 while batch b is still running (a false positive
// only delays a read).
constexpr int kDepLog = 18;
constexpr uint32_t kDepWords = 1u << (kDepLog - 5);
__device__ __forceinline__ uint32_t dep_bit(uint32_t rowid) { return hrow(rowid) >> (32 - kDepLog); }

// ---------------------------------------------------------------------------
// Kernel parameters shared by the data-phase kernels.
// ---------------------------------------------------------------------------
// Written by the pre-pass for every batch: its learning rate (FP32) and the
// salt of its stochastic rounding (sr_salt).
struct BatchParams {
    float eta;
    uint32_t salt;
};

struct DataParams {
    void* U;
    void* C;       // order 2 context table; == U for order 1
    int order, K;  // records have K+2 entries
    int apply_warps;  // warps of an apply block (batched schedule)
    int64_t n_nodes;
    uint32_t row_bits;
    const int32_t* rec;      // [chunk samples][K+2]
    const uint32_t* slot_info;  // [chunk samples][K+2]: position, or the singleton bit
    const uint4* seg;        // [n_batches][sl.cap] shared segments by class: {first position, length, row, pair count}
    const uint32_t* scount;  // [n_batches][kCounts] segments of each list
    SegLayout sl;
    float* slab;             // [batch * (K+2)][D], by position within the batch
    const uint32_t* depmap;  // [n_batches][kDepWords] rows each batch touches (bit dep_bit(row id))
    int64_t chunk_samples;
    int64_t batch;
    int n_batches;
    const BatchParams* bpar;  // [n_batches]
    float lambda, alpha_neg;
    uint32_t* status;
    // persistent schedule
    uint32_t* gbar;           // grid barrier: {arrivals, completed rounds}, zero at launch
    int slots;                // shared-memory row slots per warp (1 or 2)
    int64_t spin_limit;
    uint32_t* abort_word;
};

// Record entry idx of the group's sample: lane idx % L holds entries
// idx < L in `held`; later ones are read from memory.
__device__ __forceinline__ int32_t shfl_w(uint32_t gm, int32_t v, int src, int w) { return __shfl_sync(gm, v, src, w); }
__device__ __forceinline__ uint32_t shfl_w(uint32_t gm, uint32_t v, int src, int w) { return __shfl_sync(gm, v, src, w); }

template <int L, typename T>
__device__ __forceinline__ T rec_entry(uint32_t gm, T held, const T* row, int idx, bool active) {
    T v = shfl_w(gm, held, idx % L, L);
    if (idx >= L) v = active ? row[idx] : T{};
    return v;
}

// ---------------------------------------------------------------------------
// Per-sample work.
// ctx_stage: this warp's shared staging area, (K+1) x 32 lanes x E floats.
// ---------------------------------------------------------------------------
// The K+2 <= JB+1 record entries and places of a lane group's sample, entry i
// in lane i mod L.
template <int L, int JB>
struct Held {
    static constexpr int H = (JB + L) / L;
    int32_t r[H];
    uint32_t i[H];
    __device__ __forceinline__ void load(const DataParams& p, int64_t s_local, int lig, bool active) {
        const int R = p.K + 2;
        const int64_t at = (active ? s_local : 0) * R;
#pragma unroll
        for (int k = 0; k < H; ++k) {
            const bool in = active && k * L + lig < R;
            r[k] = in ? p.rec[at + k * L + lig] : 0;
            i[k] = in ? p.slot_info[at + k * L + lig] : 0u;
        }
    }
    __device__ __forceinline__ int32_t row(uint32_t gm, int idx) const { return __shfl_sync(gm, r[idx / L], idx % L, L); }
    __device__ __forceinline__ uint32_t place(uint32_t gm, int idx) const { return __shfl_sync(gm, i[idx / L], idx % L, L); }
};

// Register-resident gather body for K + 1 <= JB: the K+1 context rows stay in
// registers; the dots and their reductions are independent chains.  Same
// arithmetic, in the same order, as the staged body.
//
// All of a batch's warps run at once (4,096 samples at d = 128 are one wave of
// 27 warps an SM), so after the row loads arrive the gather is bound by issue
// slots: 1,960,000 warp instructions a batch were 1.6 of its 4.0 us (R-MAT 20,
// K = 5).  Hence the transposed reduction (one sigmoid per lane instead of
// K+1), packed FP32 pairs for everything but the dots (whose order over a
// lane's values is fixed), and one selected address and value per FP32 row
// instead of two branches: 1,420,000 warp instructions.  2^22 samples of one
// order in BF16: 7.80 -> 6.69 ms; both orders FP32 12.09 -> 11.75.
template <int D, int DT, int JB>
__device__ __forceinline__ void sample_body_reg(const DataParams& p, int lig, bool active, float eta, uint32_t salt,
                                                uint32_t gm, const Held<Geom<D, DT>::L, JB>& h) {
    using G = Geom<D, DT>;
    using T = Transposed<G::L, JB>;
    const int32_t u = h.row(gm, 0);
    float xu[G::E];
    float c[JB][G::E];
    load_row<D, DT>(p.U, u, lig, xu);
#pragma unroll
    for (int j = 0; j < JB; ++j) {
        const int32_t y = h.row(gm, 1 + j);
        if (j <= p.K) {
            load_row<D, DT>(p.C, y, lig, c[j]);
        } else {
#pragma unroll
            for (int e = 0; e < G::E; ++e) c[j][e] = 0.0f;
        }
    }
    float sj[JB];
#pragma unroll
    for (int j = 0; j < JB; ++j) {
        sj[j] = 0.0f;
#pragma unroll
        for (int e = 0; e < G::E; ++e) sj[j] = fmaf(xu[e], c[j][e], sj[j]);
    }
    T::reduce(sj, lig);
    float gv[T::kept()];
#pragma unroll
    for (int i = 0; i < T::kept(); ++i) {
        const float sig = 1.0f / (1.0f + expf(-sj[i]));
        gv[i] = i == 0 && (lig & T::split()) == 0 ? eta * (1.0f - sig) : -eta * p.alpha_neg * sig;
    }
    const float decay = eta * p.lambda;
    float du[G::E];
#pragma unroll
    for (int e = 0; e < G::E; ++e) du[e] = 0.0f;
#pragma unroll
    for (int j = 0; j < JB; ++j) {
        if (j > p.K) continue;
        const float g = __shfl_sync(0xFFFFFFFFu, gv[T::slot(j)], T::lane(j), G::L);
        vfma(du, g, c[j], du);
        const uint32_t inf = h.place(gm, 1 + j);
        const int32_t y = h.row(gm, 1 + j);
        const bool single = (inf & kSingleBit) != 0;
        // a singleton's new row c - decay c + g x, or the contribution g x
        float x[G::E];
        if constexpr (DT == LINE_DTYPE_F32) {
            vfma(x, -decay, c[j], c[j]);
#pragma unroll
            for (int e = 0; e < G::E; ++e) x[e] = single ? x[e] : -0.0f;  // (g x) + -0 is g x, sign of zero included
            vfma(x, g, xu, x);
            float* dst = (single ? reinterpret_cast<float*>(p.C) + (int64_t)y * D : p.slab + (int64_t)inf * D) + lig * G::E;
            if (active) {
#pragma unroll
                for (int q = 0; q < G::NV; ++q)
                    st_cg(reinterpret_cast<float4*>(dst) + q, make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]));
            }
        } else if (active) {
            if (single) {
                vfma(x, -decay, c[j], c[j]);
                vfma(x, g, xu, x);
                store_row<D, DT>(p.C, y, lig, x, salt, p.order == 2 ? 1u : 0u);
            } else {
                vmul(x, g, xu);
                float4* dst = reinterpret_cast<float4*>(p.slab + (int64_t)inf * D + lig * G::E);
#pragma unroll
                for (int q = 0; q < G::NV; ++q) st_cg(dst + q, make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]));
            }
        }
    }
    const uint32_t inf0 = h.place(gm, 0);
    if (active) {
        if (inf0 & kSingleBit) {
            vfma(xu, -((float)(p.K + 1) * decay), xu, xu);
#pragma unroll
            for (int e = 0; e < G::E; ++e) xu[e] += du[e];
            store_row<D, DT>(p.U, u, lig, xu, salt, 0u);
        } else {
            float4* dst = reinterpret_cast<float4*>(p.slab + (int64_t)inf0 * D + lig * G::E);
#pragma unroll
            for (int q = 0; q < G::NV; ++q) st_cg(dst + q, make_float4(du[4 * q], du[4 * q + 1], du[4 * q + 2], du[4 * q + 3]));
        }
    }
}

// This lane's values of row j of a set of staged rows (D values each in the
// table's type, in shared memory).
template <int D, int DT>
__device__ __forceinline__ void slot_row(const unsigned char* set, int j, int lig, float (&v)[Geom<D, DT>::E]) {
    using G = Geom<D, DT>;
    if constexpr (DT == LINE_DTYPE_F32) {
        const float4* q = reinterpret_cast<const float4*>(set + (size_t)j * D * 4 + (size_t)lig * G::E * 4);
#pragma unroll
        for (int k = 0; k < G::NV; ++k) {
            const float4 a = q[k];
            v[4 * k] = a.x;
            v[4 * k + 1] = a.y;
            v[4 * k + 2] = a.z;
            v[4 * k + 3] = a.w;
        }
    } else {
        const uint2* q = reinterpret_cast<const uint2*>(set + (size_t)j * D * 2 + (size_t)lig * G::E * 2);
#pragma unroll
        for (int k = 0; k < G::NV; ++k) {
            const uint2 a = q[k];
            v[4 * k] = __uint_as_float(a.x << 16);
            v[4 * k + 1] = __uint_as_float(a.x & 0xFFFF0000u);
            v[4 * k + 2] = __uint_as_float(a.y << 16);
            v[4 * k + 3] = __uint_as_float(a.y & 0xFFFF0000u);
        }
    }
}

// Staged gather body (any K): the K+1 context rows come into shared memory by
// asynchronous 16-byte copies past L1 (stage: (K+1) D values of the table's
// type per lane group), all in flight at once and without registers; the dots
// are reduced JB at a time.  Same arithmetic, in the same order, as the
// register body.  Rows moved through registers, four or eight at a time,
// waited for memory two or three times a sample: 2^19 samples at d = 256,
// K = 10 took 4.62 ms, like this 3.72 (BF16 4.00 and 2.98; d = 64, K = 10, B = 4096:
// 1.71 and 1.35).
template <int D, int DT>
__device__ __forceinline__ void sample_body_staged(const DataParams& p, int lig, bool active, float eta, uint32_t salt,
                                                   uint32_t gm, int32_t r0, uint32_t i0, const int32_t* rec,
                                                   const uint32_t* info, unsigned char* stage) {
    using G = Geom<D, DT>;
    constexpr int kRowBytes = D * (DT == LINE_DTYPE_F32 ? 4 : 2);
    const int32_t u = __shfl_sync(gm, r0, 0, G::L);
    for (int j = 0; j <= p.K; ++j) {
        const int32_t y = rec_entry<G::L>(gm, r0, rec, 1 + j, active);
        const unsigned char* from = reinterpret_cast<const unsigned char*>(p.C) + (int64_t)y * kRowBytes;
        for (int o = lig * 16; o < kRowBytes; o += G::L * 16) cp_async16(stage + j * kRowBytes + o, from + o);
    }
    float xu[G::E];
    load_row<D, DT>(p.U, u, lig, xu);
    cp_async_wait_all();
    __syncwarp(gm);
    const uint32_t ctx_table = p.order == 2 ? 1u : 0u;
    const float etalam = eta * p.lambda;
    float du[G::E];
#pragma unroll
    for (int e = 0; e < G::E; ++e) du[e] = 0.0f;
    constexpr int JB = 8;  // dot products reduced together
    using T = Transposed<G::L, JB>;
    for (int j0 = 0; j0 <= p.K; j0 += JB) {
        float sj[JB];
#pragma unroll
        for (int jj = 0; jj < JB; ++jj) {
            sj[jj] = 0.0f;
            if (j0 + jj <= p.K) {
                float c[G::E];
                slot_row<D, DT>(stage, j0 + jj, lig, c);
#pragma unroll
                for (int e = 0; e < G::E; ++e) sj[jj] = fmaf(xu[e], c[e], sj[jj]);
            }
        }
        T::reduce(sj, lig);
        float gv[T::kept()];
#pragma unroll
        for (int i = 0; i < T::kept(); ++i) {
            const float sig = 1.0f / (1.0f + expf(-sj[i]));
            gv[i] = i == 0 && j0 == 0 && (lig & T::split()) == 0 ? eta * (1.0f - sig) : -eta * p.alpha_neg * sig;
        }
#pragma unroll
        for (int jj = 0; jj < JB; ++jj) {
            const int j = j0 + jj;
            if (j > p.K) break;
            float c[G::E];
            slot_row<D, DT>(stage, j, lig, c);
            const float g = __shfl_sync(0xFFFFFFFFu, gv[T::slot(jj)], T::lane(jj), G::L);
            vfma(du, g, c, du);
            const uint32_t inf = rec_entry<G::L>(gm, i0, info, 1 + j, active);
            const int32_t y = rec_entry<G::L>(gm, r0, rec, 1 + j, active);
            if (active) {
                if (inf & kSingleBit) {
                    // the only reader of row y in this batch: write it now
                    vfma(c, -etalam, c, c);
                    vfma(c, g, xu, c);
                    store_row<D, DT>(p.C, y, lig, c, salt, ctx_table);
                } else {
                    vmul(c, g, xu);
                    float4* dst = reinterpret_cast<float4*>(p.slab + (int64_t)inf * D + lig * G::E);
#pragma unroll
                    for (int q = 0; q < G::E / 4; ++q) st_cg(dst + q, make_float4(c[4 * q], c[4 * q + 1], c[4 * q + 2], c[4 * q + 3]));
                }
            }
        }
    }
    const uint32_t inf0 = shfl_w(gm, i0, 0, G::L);
    if (active) {
        if (inf0 & kSingleBit) {
            const float decay = (float)(p.K + 1) * etalam;
#pragma unroll
            for (int e = 0; e < G::E; ++e) xu[e] = fmaf(-decay, xu[e], xu[e]) + du[e];
            store_row<D, DT>(p.U, u, lig, xu, salt, 0u);
        } else {
            float4* dst = reinterpret_cast<float4*>(p.slab + (int64_t)inf0 * D + lig * G::E);
#pragma unroll
            for (int q = 0; q < G::E / 4; ++q) st_cg(dst + q, make_float4(du[4 * q], du[4 * q + 1], du[4 * q + 2], du[4 * q + 3]));
        }
    }
}

// ---------------------------------------------------------------------------
// Per shared segment: fixed-order sum of its contiguous slab entries and the
// write-back.
// ---------------------------------------------------------------------------
template <int D, int DT>
__device__ __forceinline__ void segment_item(const DataParams& p, uint4 d, int lig, bool active, float eta,
                                             uint32_t salt) {
    using G = Geom<D, DT>;
    constexpr int PF = G::E <= 4 ? 8 : 4;  // slab entries in flight per lane
    if (!active) return;
    // d = {first position, length, row, pair count}
    const uint32_t len = d.y;
    const uint32_t rowid = d.z & ((1u << p.row_bits) - 1u);
    const bool is_c = p.order == 2 && rowid >= (uint32_t)p.n_nodes;
    void* table = is_c ? p.C : p.U;
    const int64_t row = is_c ? (int64_t)rowid - p.n_nodes : (int64_t)rowid;
    float x[G::E];
    load_row<D, DT>(table, row, lig, x);
    float acc[G::E];
#pragma unroll
    for (int e = 0; e < G::E; ++e) acc[e] = 0.0f;
    const float* base = p.slab + (int64_t)d.x * D + lig * G::E;
    for (uint32_t c0 = 0; c0 < len; c0 += kChunk) {
        float part[G::E];
#pragma unroll
        for (int e = 0; e < G::E; ++e) part[e] = 0.0f;
#pragma unroll
        for (uint32_t k0 = 0; k0 < kChunk; k0 += PF) {
            float4 buf[PF][G::E / 4];
#pragma unroll
            for (int kk = 0; kk < PF; ++kk) {
                if (c0 + k0 + kk < len) {
                    const float4* src = reinterpret_cast<const float4*>(base + (int64_t)(c0 + k0 + kk) * D);
#pragma unroll
                    for (int q = 0; q < G::E / 4; ++q) buf[kk][q] = ld_cg(src + q);
                }
            }
#pragma unroll
            for (int kk = 0; kk < PF; ++kk) {
                if (c0 + k0 + kk < len) {
#pragma unroll
                    for (int q = 0; q < G::E / 4; ++q) {
                        part[4 * q] += buf[kk][q].x;
                        part[4 * q + 1] += buf[kk][q].y;
                        part[4 * q + 2] += buf[kk][q].z;
                        part[4 * q + 3] += buf[kk][q].w;
                    }
                }
            }
        }
#pragma unroll
        for (int e = 0; e < G::E; ++e) acc[e] += part[e];
    }
    const float decay = (float)d.w * (eta * p.lambda);
#pragma unroll
    for (int e = 0; e < G::E; ++e) x[e] = fmaf(-decay, x[e], x[e]) + acc[e];
    store_row<D, DT>(table, row, lig, x, salt, is_c ? 1u : 0u);
}

// A shared segment of more than one chunk, summed by a team of `ts` lane
// groups of the CTA (this one is group g, member g % ts): member w
// sums chunks w, w + ts, ... (entry order within a chunk); the first member
// adds the partials in chunk order - the same order as segment_item, so the
// result does not depend on the team.  Called by all threads of the CTA, with
// the same number of rounds.  part: shared, one row of D floats per group.
template <int D, int DT>
__device__ __forceinline__ void segment_team(const DataParams& p, uint4 d, uint32_t ts, uint32_t g, int lig, float eta,
                                             uint32_t salt, float* part) {
    using G = Geom<D, DT>;
    constexpr int PF = G::E <= 4 ? 8 : 4;
    const uint32_t tg = g % ts;
    const bool first = d.y && tg == 0;
    const uint32_t rowid = d.z & ((1u << p.row_bits) - 1u);
    const bool is_c = p.order == 2 && rowid >= (uint32_t)p.n_nodes;
    float acc[G::E];
#pragma unroll
    for (int e = 0; e < G::E; ++e) acc[e] = 0.0f;
    const float* src = p.slab + ((int64_t)d.x + tg * kChunk) * D + lig * G::E;
    float* mine = part + g * D + lig * G::E;
    const uint32_t rounds = max(1u, (d.y + kChunk * ts - 1) / (kChunk * ts));
    // left: entries of the segment from this member's chunk on
    int left = (int)d.y - (int)(tg * kChunk);
    for (uint32_t r = 0; r < rounds; ++r) {
        if (left > 0) {
            float pt[G::E];
#pragma unroll
            for (int e = 0; e < G::E; ++e) pt[e] = 0.0f;
#pragma unroll
            for (int k0 = 0; k0 < (int)kChunk; k0 += PF) {
                float4 buf[PF][G::E / 4];
#pragma unroll
                for (int kk = 0; kk < PF; ++kk) {
                    if (k0 + kk < left) {
#pragma unroll
                        for (int q = 0; q < G::E / 4; ++q)
                            buf[kk][q] = ld_cg(reinterpret_cast<const float4*>(src + (k0 + kk) * D) + q);
                    }
                }
#pragma unroll
                for (int kk = 0; kk < PF; ++kk) {
                    if (k0 + kk < left) {
#pragma unroll
                        for (int q = 0; q < G::E / 4; ++q) {
                            pt[4 * q] += buf[kk][q].x;
                            pt[4 * q + 1] += buf[kk][q].y;
                            pt[4 * q + 2] += buf[kk][q].z;
                            pt[4 * q + 3] += buf[kk][q].w;
                        }
                    }
                }
            }
            float4* dst = reinterpret_cast<float4*>(mine);
#pragma unroll
            for (int q = 0; q < G::E / 4; ++q) dst[q] = make_float4(pt[4 * q], pt[4 * q + 1], pt[4 * q + 2], pt[4 * q + 3]);
        }
        __syncthreads();
        if (first) {
            const int nr = min((int)ts, (left + (int)kChunk - 1) / (int)kChunk);
#pragma unroll 4
            for (int w = 0; w < nr; ++w) {
                const float4* v4 = reinterpret_cast<const float4*>(mine + w * D);
#pragma unroll
                for (int q = 0; q < G::E / 4; ++q) {
                    const float4 v = v4[q];
                    acc[4 * q] += v.x;
                    acc[4 * q + 1] += v.y;
                    acc[4 * q + 2] += v.z;
                    acc[4 * q + 3] += v.w;
                }
            }
        }
        if (r + 1 < rounds) __syncthreads();
        left -= (int)(ts * kChunk);
        src += (int64_t)ts * kChunk * D;
    }
    if (first) {
        void* table = is_c ? p.C : p.U;
        const int64_t row = is_c ? (int64_t)rowid - p.n_nodes : (int64_t)rowid;
        float x[G::E];
        load_row<D, DT>(table, row, lig, x);
        const float decay = (float)d.w * (eta * p.lambda);
#pragma unroll
        for (int e = 0; e < G::E; ++e) x[e] = fmaf(-decay, x[e], x[e]) + acc[e];
        store_row<D, DT>(table, row, lig, x, salt, is_c ? 1u : 0u);
    }
}

// Warps of an apply block: 16 when one order trains alone (a hub row's
// chunks are summed in fewer rounds), 8 when two orders train concurrently
// (smaller blocks interleave better with the other order's kernels).
constexpr int kApplyWarpsAlone = 16, kApplyWarpsShared = 8;

// ---------------------------------------------------------------------------
// Batched schedule: one launch per phase per batch.
// ---------------------------------------------------------------------------
constexpr size_t kMaxSmem = 200 * 1024;

// Gathers run in blocks of at most 4 warps at 8 blocks per SM (at most 64
// registers), so that a 4,096-sample batch (4,096 warps at d = 128) is
// resident in one wave and still leaves registers on every SM for the
// pre-pass kernels of the next chunk (one batch at 72 registers filled 95%
// of the register file, and any pre-pass block displaced gather warps).
constexpr int kGatherWarps = 4;


// JB: context rows held in registers (K + 1 <= JB), or 0 for the staged body.
// The next kernel may start at once, and its blocks then wait on the SMs.  At
// D = 256 both kernels' blocks are small enough for those of the next two
// batches to gather there too, which held up the running ones: FP32 batches of
// up to 1,600 samples ran up to 25% longer than with larger blocks.  So at D =
// 256, and with eight rows in registers, the gather lets the apply start after
// its own wait, and at D = 256 the apply of an FP32 order that trains alone, with
// batches of up to kLateItems entries, lets the next gather start likewise.
// 2^18 samples of one order, FP32, D = 256, K = 3: R-MAT 16, B = 768 and 1,024
// 2.65 and 2.39 ms with both starts at once, 1.86 and 1.64 like this; R-MAT 18,
// K = 10, B = 1,024 and 1,500: 3.50 and 2.41, 2.71 and 2.34.  D = 128, K = 7, B =
// 900: 1.77 and 1.62.  The apply's late start costs larger FP32 batches 2% (K =
// 10, B = 2,048: 1.97 -> 2.02), BF16 ones up to 10% and two orders, which fill
// the SMs for each other, up to 13%.
constexpr int64_t kLateItems = 18432;

template <int D, int DT, int JB>
__global__ void __launch_bounds__(kGatherWarps * 32, 8) k_gather(DataParams p, int b) {
    using G = Geom<D, DT>;
    extern __shared__ float4 smem4[];
    constexpr bool kLate = D > 128 || JB == 8;
    if constexpr (!kLate) pdl_launch_dependents();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int grp = lane / G::L, lig = lane % G::L;
    const int64_t s_begin = (int64_t)b * p.batch;
    const int64_t s_end = min(s_begin + p.batch, p.chunk_samples);
    const int64_t s_local = s_begin + ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * G::GPW + grp;
    const bool active = s_local < s_end;
    const uint32_t gm = group_mask<G::L>(grp);
    // the chunk's index data comes from the pre-pass: read before the wait
    // (which has no effect without a programmatic launch)
    const BatchParams bp = p.bpar[b];
    if constexpr (JB > 0) {
        Held<G::L, JB> h;
        h.load(p, s_local, lig, active);
        pdl_wait();  // the tables' rows: written by the previous kernel
        if constexpr (kLate) pdl_launch_dependents();
        sample_body_reg<D, DT, JB>(p, lig, active, bp.eta, bp.salt, gm, h);
    } else {
        const int R = p.K + 2;
        const int64_t sbase = (active ? s_local : 0) * R;
        const int32_t* rec = p.rec + sbase;
        const uint32_t* info = p.slot_info + sbase;
        const int32_t r0 = (active && lig < R) ? rec[lig] : 0;
        const uint32_t i0 = (active && lig < R) ? info[lig] : 0u;
        pdl_wait();
        if constexpr (kLate) pdl_launch_dependents();
        unsigned char* stage = reinterpret_cast<unsigned char*>(smem4) +
                               (size_t)(warp * G::GPW + grp) * (p.K + 1) * D * (DT == LINE_DTYPE_F32 ? 4 : 2);
        sample_body_staged<D, DT>(p, lig, active, bp.eta, bp.salt, gm, r0, i0, rec, info, stage);
    }
}

// The first long_blocks() blocks take the batch's segments of several chunks,
// those after them the short ones, one per lane group; blocks that the short
// ones leave free help with the long ones, and return at once where there is
// nothing to help with (a waiting block holds registers that the next
// gather's blocks could start in: 4% of one order's time).  A block of NG
// lane groups takes one long segment, or up to NG/2, NG/4 or NG/8 of classes
// 1, 2 and 3 (a team per segment, a lane group per chunk, one round).
// Bound: latency - a slab read from L2, a sum through shared memory and the
// row's write.  On small or skewed graphs most segments are long (R-MAT 16,
// B = 4096: 320 of 5,000 a batch, 814 chunks): with one block per long
// segment, 64 of them, 2^22 samples took 12.1 ms (one order) and 17.0 (both);
// with teams 8.6 and 12.8.  R-MAT 14 at d = 64: 17.2 and 7.6; 1,024 nodes at
// d = 32: 22.2 and 8.7.  R-MAT 20: 7.33 and 7.51 (FP32), 6.54 and 6.51 (BF16),
// both orders 11.66 and 11.30.
template <int NW>
constexpr uint32_t long_blocks() {
    return 1024 / NW;
}
template <int D, int DT, int NW>
__global__ void __launch_bounds__(NW * 32, D <= 128 ? 32 / NW : 1) k_apply(DataParams p, int b) {
    using G = Geom<D, DT>;
    constexpr uint32_t kLongBlocks = long_blocks<NW>();
    constexpr uint32_t NG = NW * G::GPW, kLogNG = NG == 8 ? 3 : NG == 16 ? 4 : NG == 32 ? 5 : NG == 64 ? 6 : 7;
    static_assert(NG == 1u << kLogNG, "a block's lane groups");
    __shared__ __align__(16) float part[NG * D];
    // (see k_gather)
    const bool late = D > 128 && DT == LINE_DTYPE_F32 && p.apply_warps == kApplyWarpsAlone && p.batch * (p.K + 2) <= kLateItems;
    if (!late) pdl_launch_dependents();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int grp = lane / G::L, lig = lane % G::L;
    const uint32_t g = (uint32_t)(warp * G::GPW + grp);
    // The lists come from the pre-pass and are read before the wait, the short
    // segment without waiting for the counts: little of this prologue overlaps
    // the gather, whose blocks hold the register file.
    const uint32_t* cnt = p.scount + (size_t)b * kCounts;
    const uint4* seg = p.seg + (size_t)b * p.sl.cap;
    const uint32_t n0 = cnt[0], nl = cnt[kLong], most = p.sl.off[1];  // class 0 begins at 0
    const float eta = p.bpar[b].eta;
    const uint32_t salt = p.bpar[b].salt;
    uint32_t m = blockIdx.x >= kLongBlocks ? (blockIdx.x - kLongBlocks) * NG + g : most;
    const uint32_t first = m < most ? m : p.sl.off[kLong] + blockIdx.x;
    uint4 d = first < p.sl.cap ? seg[first] : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t nsb = min(gridDim.x - kLongBlocks, (n0 + NG - 1) / NG);  // blocks with short segments
    if (blockIdx.x - kLongBlocks < nsb) {
        pdl_wait();  // the slab and the rows: written by the gather
        if (late) pdl_launch_dependents();
        while (m < n0) {
            segment_item<D, DT>(p, d, lig, true, eta, salt);
            m += nsb * NG;
            if (m < n0) d = seg[m];
        }
        return;
    }
    // few segments of several chunks: one a block (an SM reads a segment
    // faster when it reads no other)
    if (nl <= kLongBlocks) {
        // the first block waits even without a segment: the next gather relies
        // on this kernel's end coming after the gather's
        if (blockIdx.x >= nl && blockIdx.x != 0) return;
        if (blockIdx.x >= nl) d.y = 0u;
        pdl_wait();
        segment_team<D, DT>(p, d, NG, g, lig, eta, salt, part);
        return;
    }
    const uint32_t helper = blockIdx.x < kLongBlocks ? blockIdx.x : blockIdx.x - nsb, helpers = gridDim.x - nsb;
    for (uint32_t t = helper;; t += helpers) {
        // (the counts are read again for every task: held over segment_team
        // they would not fit 64 registers)
        const uint4 n03 = ld_again(reinterpret_cast<const uint4*>(cnt));
        const uint32_t n4 = ld_again(cnt + 4);
        const uint32_t t1 = (n03.y + NG / 2 - 1) / (NG / 2), t2 = (n03.z + NG / 4 - 1) / (NG / 4),
                       t3 = (n03.w + NG / 8 - 1) / (NG / 8);
        if (t >= t1 + t2 + t3 + n4) return;  // (not the first block's first task)
        // task t, the longest segments first
        uint32_t lts = kLogNG, at = t, n = n4, off = p.sl.off[4];
        if (at >= n4) {
            at -= n4, lts = 3, n = n03.w, off = p.sl.off[3];
            if (at >= t3) {
                at -= t3, lts = 2, n = n03.z, off = p.sl.off[2];
                if (at >= t2) at -= t2, lts = 1, n = n03.y, off = p.sl.off[1];
            }
        }
        const uint32_t k = (at << (kLogNG - lts)) + (g >> lts);
        d = k < n ? seg[off + k] : make_uint4(0u, 0u, 0u, 0u);
        if (t == helper) pdl_wait();
        else __syncthreads();  // `part` is read by the last task
        segment_team<D, DT>(p, d, 1u << lts, g, lig, eta, salt, part);
    }
}

// ---------------------------------------------------------------------------
// Persistent schedule (LINE_MODE_PERSISTENT): one cooperative launch per
// chunk; one CTA of W warps per SM stays resident for all the chunk's
// batches.  For batch b:
//   gather  warp u takes the samples of units u, u + NW, ... (NW warps in
//           all; a unit is one sample per lane group).  A sample's K+2 rows
//           (U[u], then the context rows) are brought into the warp's
//           shared-memory slot by bulk copies (cp.async.bulk) that complete
//           on the slot's mbarrier; with two slots the next unit's copies run
//           while one unit is computed.  The arithmetic is the batched
//           gather's, reading the rows from shared memory; singleton rows
//           are written back, shared rows' contributions go to the slab.
//   barrier (grid-wide)
//   apply   each warp first starts the copies of its first unit of batch b+1
//           for the rows that batch b does not touch (b's row map: those rows
//           are not written in batch b); then every CTA applies some of
//           batch b's long shared segments (all its warps on one segment)
//           and every lane group some of its short ones.
//   barrier
// The rows of batch b+1 that batch b touches are copied after the second
// barrier.  Every wait is bounded: a barrier or a copy that does not finish
// within spin_limit polls records DEV_ERR_TIMEOUT, raises the abort word,
// waits (bounded) for the warp's own copies in flight, and returns.
// ---------------------------------------------------------------------------
constexpr int kPersistMaxWarps = 16;
constexpr int kPersistDefaultWarps = 16;

__device__ __forceinline__ void fail_abort(const DataParams& p) {
    atomicOr(p.status, DEV_ERR_TIMEOUT);
    atomicExch(p.abort_word, 1u);
}

// Grid-wide barrier: round r completes when all CTAs have arrived r+1 times
// (gbar[0] counts arrivals; the last arriver publishes r+1 in gbar[1]).
// Every thread's earlier global writes are visible to every CTA after it.
// Returns false when the wait ran out or another CTA aborted.
__device__ __forceinline__ bool grid_barrier(const DataParams& p, uint32_t r, uint32_t* s_flag) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        bool ok = true;
        const uint32_t old = atom_add_acq_rel(p.gbar, 1u);
        if (old == (r + 1u) * gridDim.x - 1u) {
            st_release(p.gbar + 1, r + 1u);
        } else {
            int64_t it = 0;
            while (ld_acquire(p.gbar + 1) < r + 1u) {
                if (++it > p.spin_limit || *(volatile const uint32_t*)p.abort_word) {
                    ok = false;
                    break;
                }
                if (it > 64) __nanosleep(32);
            }
        }
        if (!ok) fail_abort(p);
        *s_flag = ok ? 1u : 0u;
    }
    __syncthreads();
    return *s_flag != 0u;
}

// One lane group's sample from its staged rows (slot: row 0 = U[u], rows
// 1..K+1 = the context rows, D values each in the table's type).  The
// arithmetic is sample_body_staged's, in the same order.
template <int D, int DT>
__device__ __forceinline__ void sample_body_slot(const DataParams& p, int lig, bool active, float eta, uint32_t salt,
                                                 uint32_t gm, int32_t r0, uint32_t i0, const int32_t* rec,
                                                 const uint32_t* info, const unsigned char* set) {
    using G = Geom<D, DT>;
    constexpr int JB = 8;
    const int32_t u = __shfl_sync(gm, r0, 0, G::L);
    float xu[G::E];
    slot_row<D, DT>(set, 0, lig, xu);
    const uint32_t ctx_table = p.order == 2 ? 1u : 0u;
    const float etalam = eta * p.lambda;
    float du[G::E];
#pragma unroll
    for (int e = 0; e < G::E; ++e) du[e] = 0.0f;
    for (int j0 = 0; j0 <= p.K; j0 += JB) {
        float sj[JB];
#pragma unroll
        for (int jj = 0; jj < JB; ++jj) {
            sj[jj] = 0.0f;
            if (j0 + jj <= p.K) {
                float c[G::E];
                slot_row<D, DT>(set, 1 + j0 + jj, lig, c);
#pragma unroll
                for (int e = 0; e < G::E; ++e) sj[jj] = fmaf(xu[e], c[e], sj[jj]);
            }
        }
#pragma unroll
        for (int o = G::L / 2; o >= 1; o >>= 1)
#pragma unroll
            for (int jj = 0; jj < JB; ++jj) sj[jj] += __shfl_xor_sync(0xFFFFFFFFu, sj[jj], o);
#pragma unroll
        for (int jj = 0; jj < JB; ++jj) {
            const int j = j0 + jj;
            if (j > p.K) break;
            float c[G::E];
            slot_row<D, DT>(set, 1 + j, lig, c);
            const float sig = 1.0f / (1.0f + expf(-sj[jj]));
            const float g = j == 0 ? eta * (1.0f - sig) : -eta * p.alpha_neg * sig;
#pragma unroll
            for (int e = 0; e < G::E; ++e) du[e] = fmaf(g, c[e], du[e]);
            const uint32_t inf = rec_entry<G::L>(gm, i0, info, 1 + j, active);
            const int32_t y = rec_entry<G::L>(gm, r0, rec, 1 + j, active);
            if (active) {
                if (inf & kSingleBit) {
                    float x[G::E];
#pragma unroll
                    for (int e = 0; e < G::E; ++e) x[e] = fmaf(g, xu[e], fmaf(-etalam, c[e], c[e]));
                    store_row<D, DT>(p.C, y, lig, x, salt, ctx_table);
                } else {
                    float4* dst = reinterpret_cast<float4*>(p.slab + (int64_t)inf * D + lig * G::E);
#pragma unroll
                    for (int q = 0; q < G::E / 4; ++q)
                        st_cg(dst + q, make_float4(g * xu[4 * q], g * xu[4 * q + 1], g * xu[4 * q + 2], g * xu[4 * q + 3]));
                }
            }
        }
    }
    const uint32_t inf0 = shfl_w(gm, i0, 0, G::L);
    if (active) {
        if (inf0 & kSingleBit) {
            const float decay = (float)(p.K + 1) * etalam;
#pragma unroll
            for (int e = 0; e < G::E; ++e) xu[e] = fmaf(-decay, xu[e], xu[e]) + du[e];
            store_row<D, DT>(p.U, u, lig, xu, salt, 0u);
        } else {
            float4* dst = reinterpret_cast<float4*>(p.slab + (int64_t)inf0 * D + lig * G::E);
#pragma unroll
            for (int q = 0; q < G::E / 4; ++q) st_cg(dst + q, make_float4(du[4 * q], du[4 * q + 1], du[4 * q + 2], du[4 * q + 3]));
        }
    }
}

// Starts the bulk copies of rows j (bit j of `want`, j < K+2) of a lane
// group's sample into its row set, completing on `bar`.  arrive: this is the
// group's last issue for the slot's current phase (an arrival, with the
// bytes); otherwise only the bytes are announced.  Row j of the sample is
// U[rec[0]] for j = 0, Ctx[rec[j]] otherwise.
template <int D, int DT>
__device__ __forceinline__ void issue_rows(const DataParams& p, const int32_t* rec, int lig, uint32_t gm, int R,
                                           uint64_t want, bool arrive, unsigned char* set, uint64_t* bar) {
    using G = Geom<D, DT>;
    constexpr uint32_t kRowBytes = D * (DT == LINE_DTYPE_F32 ? 4 : 2);
    const uint32_t bytes = (uint32_t)__popcll(want) * kRowBytes;
    if (lig == 0) {
        if (arrive) mbar_arrive_expect_tx(bar, bytes);
        else if (bytes) mbar_expect_tx(bar, bytes);
    }
    __syncwarp(gm);
    for (int j = lig; j < R; j += G::L) {
        if ((want >> j) & 1ull) {
            const int32_t row = rec[j];
            const void* table = j == 0 ? p.U : p.C;
            const unsigned char* src = reinterpret_cast<const unsigned char*>(table) + (size_t)row * kRowBytes;
            bulk_load(set + (size_t)j * kRowBytes, src, kRowBytes, bar);
        }
    }
}

// A long shared segment summed by all W warps of the CTA (runtime W): warp w
// sums chunks w, w+W, ... (entry order within a chunk); warp 0 adds the
// chunk partials in chunk order, as segment_item does.  part: W x D floats.
template <int D, int DT>
__device__ __forceinline__ void long_segment_rt(const DataParams& p, uint4 d, float eta, uint32_t salt, float* part, int W) {
    using G = Geom<D, DT>;
    constexpr int PF = G::E <= 4 ? 8 : 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool mine = lane < G::L;
    const int lig = lane;
    const uint32_t len = d.y;
    const uint32_t n_chunks = (len + kChunk - 1) / kChunk;
    const uint32_t rowid = d.z & ((1u << p.row_bits) - 1u);
    const bool is_c = p.order == 2 && rowid >= (uint32_t)p.n_nodes;
    void* table = is_c ? p.C : p.U;
    const int64_t row = is_c ? (int64_t)rowid - p.n_nodes : (int64_t)rowid;
    float x[G::E];
    if (warp == 0 && mine) load_row<D, DT>(table, row, lig, x);
    float acc[G::E];
#pragma unroll
    for (int e = 0; e < G::E; ++e) acc[e] = 0.0f;
    const float* base = p.slab + (int64_t)d.x * D + (mine ? lig : 0) * G::E;
    for (uint32_t r0 = 0; r0 < n_chunks; r0 += (uint32_t)W) {
        const uint32_t c = r0 + (uint32_t)warp;
        if (mine && c < n_chunks) {
            float pt[G::E];
#pragma unroll
            for (int e = 0; e < G::E; ++e) pt[e] = 0.0f;
            const uint32_t c0 = c * kChunk;
#pragma unroll
            for (uint32_t k0 = 0; k0 < kChunk; k0 += PF) {
                float4 buf[PF][G::E / 4];
#pragma unroll
                for (int kk = 0; kk < PF; ++kk)
                    if (c0 + k0 + kk < len)
#pragma unroll
                        for (int q = 0; q < G::E / 4; ++q)
                            buf[kk][q] = ld_cg(reinterpret_cast<const float4*>(base + (int64_t)(c0 + k0 + kk) * D) + q);
#pragma unroll
                for (int kk = 0; kk < PF; ++kk)
                    if (c0 + k0 + kk < len)
#pragma unroll
                        for (int q = 0; q < G::E / 4; ++q) {
                            pt[4 * q] += buf[kk][q].x;
                            pt[4 * q + 1] += buf[kk][q].y;
                            pt[4 * q + 2] += buf[kk][q].z;
                            pt[4 * q + 3] += buf[kk][q].w;
                        }
            }
#pragma unroll
            for (int e = 0; e < G::E; ++e) part[warp * D + lig * G::E + e] = pt[e];
        }
        __syncthreads();
        if (warp == 0 && mine) {
            const uint32_t nr = min((uint32_t)W, n_chunks - r0);
            for (uint32_t w = 0; w < nr; ++w)
#pragma unroll
                for (int e = 0; e < G::E; ++e) acc[e] += part[w * D + lig * G::E + e];
        }
        __syncthreads();
    }
    if (warp == 0 && mine) {
        const float decay = (float)d.w * (eta * p.lambda);
#pragma unroll
        for (int e = 0; e < G::E; ++e) x[e] = fmaf(-decay, x[e], x[e]) + acc[e];
        store_row<D, DT>(table, row, lig, x, salt, is_c ? 1u : 0u);
    }
}

// Row bytes of one lane group's sample set, rounded up to 128.
__host__ __device__ inline size_t persist_set_bytes(int dim, int dtype, int K) {
    return (((size_t)(K + 2) * dim * (dtype == LINE_DTYPE_F32 ? 4 : 2)) + 127) & ~(size_t)127;
}

// Dynamic shared memory of a W-warp CTA: the warps' row slots, the long
// segments' partials (W x D floats) and two mbarriers per warp.
__host__ __device__ inline size_t persist_smem_bytes(int dim, int dtype, int K, int W, int slots, int gpw) {
    return (size_t)W * slots * gpw * persist_set_bytes(dim, dtype, K) + (size_t)W * dim * sizeof(float) +
           (size_t)W * 2 * sizeof(uint64_t);
}

template <int D, int DT>
__global__ void __launch_bounds__(kPersistMaxWarps * 32, 1) k_persistent(DataParams p) {
    using G = Geom<D, DT>;
    extern __shared__ __align__(128) unsigned char psm[];
    __shared__ uint32_t s_flag;
    const int W = (int)(blockDim.x >> 5);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int grp = lane / G::L, lig = lane % G::L;
    const uint32_t gm = group_mask<G::L>(grp);
    const int R = p.K + 2;
    const size_t set_bytes = persist_set_bytes(D, DT, p.K);
    const int slots = p.slots;
    unsigned char* wslots = psm + (size_t)warp * slots * G::GPW * set_bytes;
    float* part = reinterpret_cast<float*>(psm + (size_t)W * slots * G::GPW * set_bytes);
    uint64_t* bars = reinterpret_cast<uint64_t*>(part + (size_t)W * D) + 2 * warp;
    if (lane == 0) {
        mbar_init(bars, G::GPW);  // one arrival per lane group and phase
        mbar_init(bars + 1, G::GPW);
        mbar_init_fence();
    }
    __syncwarp();
    const int64_t NW = (int64_t)gridDim.x * W;                 // warps in all
    const int64_t uwarp = (int64_t)blockIdx.x * W + warp;      // this warp
    uint32_t par0 = 0, par1 = 0;                               // phase parity of each slot
    bool pending0 = false, pending1 = false;                   // copies issued, not yet waited for
    uint64_t pre_want = 0;                                     // rows of unit 0 already requested (prefetch)
    bool prefetched = false;
    uint32_t round = 0;
    bool ok = true;
    const uint64_t all_rows = R >= 64 ? ~0ull : ((1ull << R) - 1ull);
    for (int b = 0; b < p.n_batches && ok; ++b) {
        const int64_t s_begin = (int64_t)b * p.batch;
        const int64_t nb = min((int64_t)p.batch, p.chunk_samples - s_begin);
        const int64_t units = (nb + G::GPW - 1) / G::GPW;
        const float eta = p.bpar[b].eta;
        const uint32_t salt = p.bpar[b].salt;
        const int64_t n_mine = uwarp < units ? (units - 1 - uwarp) / NW + 1 : 0;
        // ---- gather of batch b
        // copies of the first two units (unit 0's prefetched rows are in flight)
        for (int k = 0; k < 2 && k < n_mine; ++k) {
            const int64_t s_local = s_begin + (uwarp + k * NW) * G::GPW + grp;
            const bool active = s_local < s_begin + nb;
            const int32_t* rec = p.rec + (active ? s_local : 0) * R;
            uint64_t want = active ? all_rows : 0ull;
            if (k == 0 && prefetched) want &= ~pre_want;
            fence_proxy_async_global();
            issue_rows<D, DT>(p, rec, lig, gm, R, want, true, wslots + (size_t)k * G::GPW * set_bytes + grp * set_bytes,
                              bars + k);
            if (k == 0) pending0 = true;
            else pending1 = true;
        }
        prefetched = false;
        for (int64_t k = 0; k < n_mine && ok; ++k) {
            const int sl = (int)(k & 1);
            const int64_t s_local = s_begin + (uwarp + k * NW) * G::GPW + grp;
            const bool active = s_local < s_begin + nb;
            // wait for the unit's rows
            uint64_t* bar = bars + sl;
            const uint32_t par = sl ? par1 : par0;
            int64_t it = 0;
            while (!mbar_try_wait(bar, par)) {
                if (++it > p.spin_limit || *(volatile const uint32_t*)p.abort_word) {
                    ok = false;
                    break;
                }
            }
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            if (sl) {
                par1 ^= 1u;
                pending1 = false;
            } else {
                par0 ^= 1u;
                pending0 = false;
            }
            const unsigned char* set = wslots + (size_t)sl * G::GPW * set_bytes + grp * set_bytes;
            const int64_t sbase = (active ? s_local : 0) * R;
            const int32_t* rec = p.rec + sbase;
            const uint32_t* info = p.slot_info + sbase;
            const int32_t r0 = (active && lig < R) ? rec[lig] : 0;
            const uint32_t i0 = (active && lig < R) ? info[lig] : 0u;
            sample_body_slot<D, DT>(p, lig, active, eta, salt, gm, r0, i0, rec, info, set);
            // the slot's rows are read: it may be refilled by bulk copies
            fence_proxy_async_smem();
            __syncwarp();
            if (k + 2 < n_mine) {
                const int64_t s2 = s_begin + (uwarp + (k + 2) * NW) * G::GPW + grp;
                const bool act2 = s2 < s_begin + nb;
                issue_rows<D, DT>(p, p.rec + (act2 ? s2 : 0) * R, lig, gm, R, act2 ? all_rows : 0ull, true,
                                  wslots + (size_t)sl * G::GPW * set_bytes + grp * set_bytes, bar);
                if (sl) pending1 = true;
                else pending0 = true;
            }
        }
        if (!__all_sync(0xFFFFFFFFu, ok)) ok = false;
        if (!ok) {
            if (lane == 0) fail_abort(p);
            break;
        }
        if (!grid_barrier(p, round++, &s_flag)) {
            ok = false;
            break;
        }
        // ---- apply of batch b; first the prefetch of batch b+1's rows that
        // batch b does not touch
        if (b + 1 < p.n_batches) {
            const int64_t s1_begin = (int64_t)(b + 1) * p.batch;
            const int64_t nb1 = min((int64_t)p.batch, p.chunk_samples - s1_begin);
            const int64_t units1 = (nb1 + G::GPW - 1) / G::GPW;
            if (uwarp < units1) {
                const int64_t s_local = s1_begin + uwarp * G::GPW + grp;
                const bool active = s_local < s1_begin + nb1;
                const int32_t* rec = p.rec + (active ? s_local : 0) * R;
                // rows of the group's sample that batch b does not touch
                bool free_row = false;
                if (active && lig < R) {
                    const uint32_t rowid = (uint32_t)rec[lig] + (lig > 0 && p.order == 2 ? (uint32_t)p.n_nodes : 0u);
                    const uint32_t db = dep_bit(rowid);
                    free_row = !((__ldcg(p.depmap + (size_t)b * kDepWords + (db >> 5)) >> (db & 31u)) & 1u);
                }
                uint32_t fm = __ballot_sync(0xFFFFFFFFu, free_row);
                fm = G::L == 32 ? fm : (fm >> (grp * G::L)) & ((1u << G::L) - 1u);
                pre_want = (uint64_t)fm;  // rows >= L: copied after the barrier
                fence_proxy_async_global();
                issue_rows<D, DT>(p, rec, lig, gm, R, pre_want, false, wslots + grp * set_bytes, bars);
                prefetched = true;
                pending0 = true;
            }
        }
        {
            // segments of several chunks: one CTA each
            const uint32_t* cnt = p.scount + (size_t)b * kCounts;
            const uint4* seg = p.seg + (size_t)b * p.sl.cap;
            uint32_t l = blockIdx.x;
            for (int c = 1; c < kClasses; ++c) {
                for (; l < cnt[c]; l += gridDim.x)
                    long_segment_rt<D, DT>(p, seg[p.sl.off[c] + l], eta, salt, part, W);
                l -= cnt[c];
            }
            // short ones: one lane group each
            for (int64_t m = uwarp * G::GPW + grp; m < cnt[0]; m += NW * G::GPW)
                segment_item<D, DT>(p, seg[m], lig, true, eta, salt);
        }
        if (!grid_barrier(p, round++, &s_flag)) {
            ok = false;
            break;
        }
    }
    if (!ok) {
        // wait (bounded) for this warp's copies still in flight, then return
        for (int sl = 0; sl < 2; ++sl) {
            if (!(sl ? pending1 : pending0)) continue;
            uint64_t* bar = bars + sl;
            const uint32_t par = sl ? par1 : par0;
            for (int64_t it = 0; it <= p.spin_limit && !mbar_try_wait(bar, par); ++it) {
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Pre-pass kernels.
// ---------------------------------------------------------------------------
struct PrepassParams {
    const int32_t* src;
    const int32_t* dst;
    const uint2* edge_tab;
    const uint2* neg_tab;
    int64_t n_arcs, n_nodes;
    uint64_t seed;
    uint64_t t_chunk;
    int64_t chunk_samples;
    int64_t batch;
    int K, order;
    int walk;  // 1: slots 0 and 1 come from the walk sampler (no arc draw here)
    int32_t* rec;
    // per batch of the chunk (minibatch schedules): its parameters, and the
    // counters of the grouping, zeroed here
    int n_batches;
    float lr0, lr_floor;
    int lr_schedule;
    uint64_t lr_total;
    BatchParams* bpar;  // null: no per-batch outputs (Hogwild schedule)
    uint32_t* scount;
    uint32_t* pcount;
};

__device__ __forceinline__ uint64_t make_item(uint32_t rowid, uint32_t s_local, uint32_t slot) {
    return ((uint64_t)rowid << 32) | ((s_local << kSlotBits) | slot);
}

// eta of the batch starting at global sample t0: lr0 (schedule 0) or
// lr0 * max(1 - t0/T, floor) (schedule 1), in FP32, 1 - t0/T as (T - t0) / T
// from the exact integer difference.
__device__ __forceinline__ float batch_eta(const PrepassParams& p, uint64_t t0) {
    float f = 1.0f;
    if (p.lr_schedule == 1) {
        f = t0 >= p.lr_total ? 0.0f : (float)(p.lr_total - t0) / (float)p.lr_total;
        if (f < p.lr_floor) f = p.lr_floor;
    }
    return p.lr0 * f;
}

__global__ void k_chunk_draws(PrepassParams p) {
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    if (p.bpar)
        for (uint32_t b = tid; b < (uint32_t)p.n_batches; b += stride) {
            const uint64_t t0 = p.t_chunk + (uint64_t)b * (uint64_t)p.batch;
            p.bpar[b] = BatchParams{batch_eta(p, t0), sr_salt(p.seed, t0)};
            for (int k = 0; k < kCounts; ++k) p.scount[(size_t)b * kCounts + k] = 0u;
            p.pcount[b] = 0u;
        }
    const uint32_t C1 = (uint32_t)p.K + 1u, R = (uint32_t)p.K + 2u;
    const uint32_t total = (uint32_t)p.chunk_samples * C1;
    for (uint32_t q = tid; q < total; q += stride) {
        const uint32_t s = q / C1;
        const uint32_t c = q - s * C1;
        const uint4 w = draw_words(p.seed, 0u, p.t_chunk + (uint64_t)s, c);
        const uint32_t base = s * R;
        if (c == 0) {
            if (p.walk) continue;
            const uint32_t e = alias_pick(p.edge_tab, (uint64_t)p.n_arcs, w);
            p.rec[base] = __ldg(p.src + e);
            p.rec[base + 1] = __ldg(p.dst + e);
        } else {
            p.rec[base + 1 + c] = (int32_t)alias_pick(p.neg_tab, (uint64_t)p.n_nodes, w);
        }
    }
}

// ---------------------------------------------------------------------------
// Grouping of each batch's items by row.  Items of batch b occupy positions
// [b B (K+2), b B (K+2) + nb (K+2)) of the chunk, in (sample, slot) order.
// ---------------------------------------------------------------------------
constexpr int kBuckets = 256;            // bucket = 8-bit multiplicative hash of the row id

constexpr int kBucketThreads = 1024;
constexpr int kBucketWarps = kBucketThreads / 32;
constexpr uint32_t kPartItems = 16384;   // items of a batch per bucketing CTA
constexpr int kSortThreads = 256;        // one warp per bucket

struct GroupParams {
    int n_batches;
    int64_t batch;
    int64_t chunk_samples;
    uint32_t R, K, parts;  // parts: bucketing CTAs per batch
    uint32_t R_magic;       // floor(2^32 / R) + 1: i / R = mulhi(i, R_magic) for i < 2^32 / R
    uint32_t ctx_off;       // row id of the context table's first row
    const int32_t* rec;     // draws, (sample, slot) order
    uint64_t* bucketed;     // items grouped by bucket within each batch (k_group_parts: keys that exceed a CTA)
    uint64_t* tmp;          // scratch of the same size
    uint32_t* gcnt;         // [n_batches][parts][256] bucket counts of each part
    uint32_t* boff;         // [n_batches][257] bucket starts within the batch
    uint32_t* pcount;       // [n_batches] positions handed out (k_group_parts)
    // outputs
    uint32_t* slot_info;
    uint4* seg;
    uint32_t* scount;
    SegLayout sl;
    uint32_t* depmap;     // [n_batches][kDepWords] rows each batch touches (zeroed before), or null
};

__device__ __forceinline__ void batch_range(const GroupParams& q, int b, uint64_t* base, uint32_t* n) {
    const int64_t nb = min(q.batch, q.chunk_samples - (int64_t)b * q.batch);
    *base = (uint64_t)b * (uint64_t)q.batch * q.R;
    *n = (uint32_t)nb * q.R;
}

// Entry i of the chunk as an item: row id << 32 | (sample, slot).
__device__ __forceinline__ uint64_t item_at(const GroupParams& q, uint64_t at) {
    const uint32_t i = (uint32_t)at, s = i / q.R, slot = i - s * q.R;  // a chunk has fewer than 2^31 entries
    return make_item((uint32_t)q.rec[i] + (slot ? q.ctx_off : 0u), s, slot);
}

__global__ void __launch_bounds__(kBucketThreads) k_bucket_count(GroupParams q) {
    __shared__ uint32_t cnt[kBuckets];
    const int part = blockIdx.x, b = blockIdx.y;
    if (threadIdx.x < kBuckets) cnt[threadIdx.x] = 0;
    __syncthreads();
    uint64_t base;
    uint32_t n;
    batch_range(q, b, &base, &n);
    const uint32_t lo = min(n, (uint32_t)part * kPartItems), hi = min(n, lo + kPartItems);
    for (uint32_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        const uint32_t rowid = (uint32_t)(item_at(q, base + i) >> 32);
        atomicAdd(&cnt[bucket_of(rowid)], 1u);
        if (q.depmap) {
            const uint32_t db = dep_bit(rowid);
            atomicOr(q.depmap + (size_t)b * kDepWords + (db >> 5), 1u << (db & 31u));
        }
    }
    __syncthreads();
    if (threadIdx.x < kBuckets) q.gcnt[((size_t)b * q.parts + part) * kBuckets + threadIdx.x] = cnt[threadIdx.x];
}

// Stable scatter of one part: bucket start + the earlier parts' counts + the
// earlier warps' counts + the rank within the warp's rounds.
__global__ void __launch_bounds__(kBucketThreads) k_bucket_scatter(GroupParams q) {
    __shared__ uint32_t bstart[kBuckets], poff[kBuckets];
    __shared__ uint32_t wcnt[kBucketWarps][kBuckets];
    const int part = blockIdx.x, b = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t base;
    uint32_t n;
    batch_range(q, b, &base, &n);
    for (int i = threadIdx.x; i < kBucketWarps * kBuckets; i += blockDim.x) (&wcnt[0][0])[i] = 0;
    if (threadIdx.x < kBuckets) {
        const uint32_t d = threadIdx.x;
        uint32_t tot = 0, before = 0;
        for (uint32_t pp = 0; pp < q.parts; ++pp) {
            const uint32_t c = q.gcnt[((size_t)b * q.parts + pp) * kBuckets + d];
            if (pp < (uint32_t)part) before += c;
            tot += c;
        }
        bstart[d] = tot;
        poff[d] = before;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t run = 0;
        for (int d = 0; d < kBuckets; ++d) {
            const uint32_t c = bstart[d];
            bstart[d] = run;
            run += c;
        }
    }
    __syncthreads();
    if (part == 0 && threadIdx.x <= kBuckets) q.boff[(size_t)b * (kBuckets + 1) + threadIdx.x] = threadIdx.x < kBuckets ? bstart[threadIdx.x] : n;
    const uint32_t lo = min(n, (uint32_t)part * kPartItems), hi = min(n, lo + kPartItems);
    const uint32_t per = (hi - lo + kBucketWarps - 1) / kBucketWarps;
    const uint32_t wlo = min(hi, lo + warp * per), whi = min(hi, wlo + per);
    const uint32_t lt = (1u << lane) - 1u;
    for (uint32_t r = wlo; r < whi; r += 32) {
        const uint32_t i = r + lane;
        const bool valid = i < whi;
        const uint32_t d = valid ? bucket_of((uint32_t)(item_at(q, base + i) >> 32)) : 0xFFFFu;
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
        if (valid && (peers & lt) == 0) wcnt[warp][d] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x < kBuckets) {
        uint32_t run = 0;
        for (int w = 0; w < kBucketWarps; ++w) {
            const uint32_t c = wcnt[w][threadIdx.x];
            wcnt[w][threadIdx.x] = run;
            run += c;
        }
    }
    __syncthreads();
    for (uint32_t r = wlo; r < whi; r += 32) {
        const uint32_t i = r + lane;
        const bool valid = i < whi;
        const uint64_t it = valid ? item_at(q, base + i) : 0ull;
        const uint32_t d = valid ? bucket_of((uint32_t)(it >> 32)) : 0xFFFFu;
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
        const uint32_t before = valid ? wcnt[warp][d] : 0u;
        if (valid) q.bucketed[base + bstart[d] + poff[d] + before + __popc(peers & lt)] = it;
        __syncwarp();
        if (valid && (peers & lt) == 0) wcnt[warp][d] = before + __popc(peers);
        __syncwarp();
    }
}

// One stable 8-bit LSD pass of a warp over n items (global memory), by bits
// [shift, shift + 8) of the hashed row id.  cnt: the warp's 256 shared counters.
__device__ void warp_radix_pass(const uint64_t* src, uint64_t* dst, uint32_t n, uint32_t shift, uint32_t* cnt) {
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    for (int i = lane; i < kBuckets; i += 32) cnt[i] = 0;
    __syncwarp();
    for (uint32_t r = 0; r < n; r += 32) {
        const uint32_t i = r + lane;
        const bool valid = i < n;
        const uint32_t d = valid ? (hrow((uint32_t)(src[i] >> 32)) >> shift) & 255u : 0xFFFFu;
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
        if (valid && (peers & lt) == 0) cnt[d] += __popc(peers);
        __syncwarp();
    }
    // exclusive scan of the 256 counters: lane l owns counters 8l .. 8l+7
    uint32_t own = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) own += cnt[lane * 8 + k];
    uint32_t incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += v;
    }
    uint32_t run = incl - own;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t c = cnt[lane * 8 + k];
        cnt[lane * 8 + k] = run;
        run += c;
    }
    __syncwarp();
    for (uint32_t r = 0; r < n; r += 32) {
        const uint32_t i = r + lane;
        const bool valid = i < n;
        const uint64_t it = valid ? src[i] : 0ull;
        const uint32_t d = valid ? (hrow((uint32_t)(it >> 32)) >> shift) & 255u : 0xFFFFu;
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
        const uint32_t before = valid ? cnt[d] : 0u;
        if (valid) dst[before + __popc(peers & lt)] = it;
        __syncwarp();
        if (valid && (peers & lt) == 0) cnt[d] = before + __popc(peers);
        __syncwarp();
    }
}

constexpr uint32_t kWarpSortCap = 512;  // bucket sizes ranked directly in shared memory
constexpr int kSortBucketsPerCta = kSortThreads / 32;

// One warp per (bucket, batch): sort the bucket's items by row (stable), then
// find its segments.  Small buckets: a bitonic sort of (row, index) in shared
// memory; large ones: LSD radix passes in global memory.
__global__ void __launch_bounds__(kSortThreads) k_bucket_sort(GroupParams q) {
    extern __shared__ uint64_t sbuf[];  // per warp: 2 x kWarpSortCap items
    __shared__ uint32_t wcnt[kSortBucketsPerCta][kBuckets];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d = blockIdx.x * kSortBucketsPerCta + warp, b = blockIdx.y;
    if (b >= q.n_batches || d >= kBuckets) return;
    uint64_t base;
    uint32_t n;
    batch_range(q, b, &base, &n);
    const uint32_t lo = q.boff[(size_t)b * (kBuckets + 1) + d], hi = q.boff[(size_t)b * (kBuckets + 1) + d + 1];
    const uint32_t c = hi - lo;
    if (c == 0) return;
    const uint64_t* a;
    if (c <= kWarpSortCap) {
        // bitonic sort of the unique keys (hrow(row) << 32 | index) over the
        // next power of two, padded with the largest key; then items by rank
        uint64_t* in = sbuf + (size_t)warp * 2 * kWarpSortCap;
        uint64_t* key = in + kWarpSortCap;
        uint32_t P = 32;
        while (P < c) P <<= 1;
        for (uint32_t i = lane; i < P; i += 32) {
            if (i < c) {
                const uint64_t it = q.bucketed[base + lo + i];
                in[i] = it;
                key[i] = ((uint64_t)hrow((uint32_t)(it >> 32)) << 32) | i;
            } else {
                key[i] = ~0ull;
            }
        }
        __syncwarp();
        for (uint32_t kk = 2; kk <= P; kk <<= 1) {
            for (uint32_t jj = kk >> 1; jj > 0; jj >>= 1) {
                for (uint32_t t = lane; t < P / 2; t += 32) {
                    const uint32_t i = ((t & ~(jj - 1)) << 1) | (t & (jj - 1));
                    const uint32_t l = i + jj;
                    const uint64_t x = key[i], y = key[l];
                    if ((x > y) == ((i & kk) == 0)) {
                        key[i] = y;
                        key[l] = x;
                    }
                }
                __syncwarp();
            }
        }
        // sorted items replace the keys in place (each lane reads, then writes, its own slots)
        for (uint32_t r = lane; r < c; r += 32) {
            const uint64_t it = in[(uint32_t)key[r]];
            key[r] = it;
        }
        __syncwarp();
        a = key;
    } else {  // a large bucket (a very skewed draw): radix passes over the hashed row
        uint64_t* x = q.bucketed + base + lo;
        uint64_t* y = q.tmp + base + lo;
        for (uint32_t sh = 0; sh < 32; sh += 8) {
            warp_radix_pass(x, y, c, sh, wcnt[warp]);
            uint64_t* t = x;
            x = y;
            y = t;
        }
        __syncwarp();
        a = x;
    }
    const uint32_t gpos = lo;  // position of the bucket's first item in the batch
    for (uint32_t i = lane; i < c; i += 32) {
        const uint32_t key = (uint32_t)(a[i] >> 32);
        if (i > 0 && (uint32_t)(a[i - 1] >> 32) == key) continue;
        uint32_t j = i + 1;
        while (j < c && (uint32_t)(a[j] >> 32) == key) ++j;
        const uint32_t len = j - i;
        const uint32_t head = (uint32_t)(gpos + i);
        uint32_t cnt = 0;
        for (uint32_t k = i; k < j; ++k) {
            const uint32_t v = (uint32_t)a[k];
            const uint32_t slot = v & kSlotMask;
            cnt += slot == 0 ? q.K + 1 : 1u;
            const uint32_t pos = (uint32_t)(gpos + k);
            q.slot_info[(v >> kSlotBits) * q.R + slot] = len == 1 ? kSingleBit : pos;
        }
        if (len > 1) {
            const int c = seg_class(len);
            const uint32_t m = atomicAdd(q.scount + (size_t)b * kCounts + c, 1u);
            uint4* seg = q.seg + (size_t)b * q.sl.cap;
            seg[q.sl.off[c] + m] = make_uint4(head, len, key, cnt);
            if (c) seg[q.sl.off[kLong] + atomicAdd(q.scount + (size_t)b * kCounts + kLong, 1u)] = make_uint4(head, len, key, cnt);
        }
    }
}

// ---- Grouping of a batch by P = 2^log_parts independent CTAs (batches of up
// to 16 x 16,384 items).  CTA `me` of batch b owns the rows whose hrow starts
// with the bits `me`: it scans all of the batch's record entries (they are in
// L2) and keeps its own, so no CTA waits for another.
//   1. A row that occurs once needs no position: two bitmaps of 2^17 bits,
//      indexed by hrow, record which bits are hit and which are hit twice.
//      On R-MAT 20 73% of a batch's items are such rows; they (but for about
//      one in ten, which shares its bit) get the singleton mark at once.
//   2. The other items ("candidates") are counted into 4,096 sub-buckets by
//      further hrow bits and placed there as keys (hrow(row) << 32 | sample,
//      slot), in no particular order.
//   3. One thread per key compares it with the keys of its sub-bucket (about
//      three): the keys of smaller rows, of its own row, and those of its row
//      that come before it give its position, its segment's head and length.
//      Nothing is sorted.  Only a sub-bucket of more than kRankMax keys (a
//      hub row) is sorted, by one warp.
// Positions are unique within the batch and contiguous per row, in (sample,
// slot) order; where a part begins depends on the order in which the parts
// arrive, which no result depends on.
// Bound: issue slots and the latency of the three scans.  A chunk of 64
// batches of 28,672 items (R-MAT 20, d = 128, K = 5) takes 31 us with nothing
// beside it and 32 beside the data phase, on 128 CTAs (36 and 38-41 with 1,024
// sub-buckets and a reservation of list places per warp and round); the
// earlier form, which sorted all items of a batch in an 8-CTA cluster, 107 and
// 118 on 512.  16 batches of 114,688 items (8 parts each): 78 us against 276
// for the three kernels below.  One order at B = 4096 went from 8.74 to 7.80 ms for
// 2^22 samples (BF16), both orders from 13.99 to 12.09 (FP32).  Beyond 16
// parts every part's scan of the whole batch costs more than it saves.
constexpr int kPartThreads = 1024;
constexpr uint32_t kPartItems2 = 16384;  // a part's share of the items, at most
constexpr uint32_t kPartCap = 15360;     // keys held in shared memory; more go to the scratch array
constexpr int kPartMaxLog = 4;
constexpr int kLogSub = 12;
constexpr int kPartSub = 1 << kLogSub;   // sub-buckets of a part (four per thread)
constexpr uint32_t kFound = 1u << (17 - 5 + 1);  // results kept in the bitmaps' place
constexpr uint32_t kMapBits = 17;
constexpr uint32_t kRankMax = 128;

// In-place ascending sort of a[0 .. n) by one warp: a bitonic network whose
// comparators all put the minimum first (per merge size k the mirror
// comparator (i, k-1-i) within each k-block, then half-cleaners of strides
// k/4 .. 1); positions >= n act as +infinity, so comparators reaching past n
// are skipped.
__device__ __forceinline__ void warp_sort_keys(uint64_t* a, uint32_t n) {
    const int lane = threadIdx.x & 31;
    uint32_t N = 1;
    while (N < n) N <<= 1;
    for (uint32_t k = 2; k <= N; k <<= 1) {
        const uint32_t lh = 31 - __clz(k >> 1);
        for (uint32_t t = lane; t < N / 2; t += 32) {
            const uint32_t blk = t >> lh, off = t & ((k >> 1) - 1);
            const uint32_t i = blk * k + off, j = blk * k + k - 1 - off;
            if (j < n) {
                const uint64_t x = a[i], y = a[j];
                if (x > y) {
                    a[i] = y;
                    a[j] = x;
                }
            }
        }
        __syncwarp();
        for (uint32_t jj = k >> 2; jj > 0; jj >>= 1) {
            for (uint32_t t = lane; t < N / 2; t += 32) {
                const uint32_t i = ((t & ~(jj - 1)) << 1) | (t & (jj - 1)), j = i + jj;
                if (j < n) {
                    const uint64_t x = a[i], y = a[j];
                    if (x > y) {
                        a[i] = y;
                        a[j] = x;
                    }
                }
            }
            __syncwarp();
        }
    }
}

// Lists the shared segments of the warp's lanes with len > 1 (head: first
// position, z: its source entries).  Called by whole warps.
__device__ __forceinline__ void list_segments(const GroupParams& q, int b, bool is_head, uint32_t head, uint32_t len,
                                              uint32_t hv, uint32_t z) {
    const int lane = threadIdx.x & 31;
    const bool m = is_head && len > 1;
    if (!__any_sync(0xFFFFFFFFu, m)) return;
    const int cls = m ? seg_class(len) : kClasses + 1;
    // lane c reserves the places of list c
    const uint32_t longs = __ballot_sync(0xFFFFFFFFu, m && cls > 0);
    uint32_t peers = 0, count = lane == kLong ? __popc(longs) : 0u, base = 0;
#pragma unroll
    for (int c = 0; c < kClasses; ++c) {
        const uint32_t mk = __ballot_sync(0xFFFFFFFFu, cls == c);
        if (cls == c) peers = mk;
        if (lane == c) count = __popc(mk);
    }
    if (count) base = atomicAdd(q.scount + (size_t)b * kCounts + lane, count);
    const uint32_t lbase = __shfl_sync(0xFFFFFFFFu, base, kLong);
    base = __shfl_sync(0xFFFFFFFFu, base, cls);
    // pair count: K + 1 for a source entry, 1 otherwise
    if (m) {
        const uint32_t lt = (1u << lane) - 1u;
        const uint4 d = make_uint4(head, len, unhrow(hv), len + z * q.K);
        uint4* seg = q.seg + (size_t)b * q.sl.cap;
        seg[q.sl.off[cls] + base + __popc(peers & lt)] = d;
        if (cls > 0) seg[q.sl.off[kLong] + lbase + __popc(longs & lt)] = d;
    }
}

// Steps 2b and 3 for the part's nc keys, grouped by sub-bucket in a (shared
// memory, or the scratch array; inlined for each).  found: room for kFound
// results (the bitmaps, no longer needed): with at most so many keys the
// segments are counted first, and listed after one reservation of the part's
// places (a reservation per warp and round costs a round trip to L2 each).
__device__ __forceinline__ void group_segments(const GroupParams& q, const uint64_t* a, uint64_t* aw, uint32_t nc,
                                               const uint32_t* start, int log_parts, uint32_t pbase, int b,
                                               const uint16_t* big, uint32_t nbig, uint32_t* found, uint32_t* lcnt) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool later = nc <= kFound;
    for (uint32_t i0 = warp * 32; i0 < nc; i0 += kPartThreads) {
        const uint32_t i = i0 + lane;
        bool mine = i < nc;
        const uint64_t key = mine ? a[i] : 0ull;
        const uint32_t hv = (uint32_t)(key >> 32), v = (uint32_t)key;
        const uint32_t sub = (hv << log_parts) >> (32 - kLogSub);
        const uint32_t s0 = start[sub], c = start[sub + 1] - s0;
        mine = mine && c <= kRankMax;
        uint32_t lower = 0, same = 0, before = 0, z = 0;
        if (mine) {
            for (uint32_t j = 0; j < c; ++j) {
                const uint64_t k2 = a[s0 + j];
                const uint32_t h2 = (uint32_t)(k2 >> 32), v2 = (uint32_t)k2;
                lower += h2 < hv;
                if (h2 == hv) {
                    ++same;
                    before += v2 < v;
                    z += (v2 & kSlotMask) == 0;
                }
            }
        }
        const uint32_t head = pbase + s0 + lower;
        if (mine) q.slot_info[(v >> kSlotBits) * q.R + (v & kSlotMask)] = same == 1 ? kSingleBit : head + before;
        const bool is_head = mine && before == 0;
        if (later) {
            // lower, same, z <= kRankMax = 2^7: 8 bits each
            const bool m = is_head && same > 1;
            if (i < nc) found[i] = m ? (1u << 31) | (lower << 16) | (same << 8) | z : 0u;
            const int cls = m ? seg_class(same) : kClasses + 1;
#pragma unroll
            for (int cc = 0; cc < kClasses; ++cc) {
                const uint32_t mk = __ballot_sync(0xFFFFFFFFu, cls == cc);
                if (mk && lane == 0) atomicAdd(lcnt + cc, (uint32_t)__popc(mk));
            }
        } else {
            list_segments(q, b, is_head, head, same, hv, z);
        }
    }
    if (later) {
        __syncthreads();
        if (warp == 0) {
            // lane c reserves the part's places of list c
            uint32_t n = lane < kClasses ? lcnt[lane] : 0u;
            const uint32_t longs = __reduce_add_sync(0xFFFFFFFFu, lane > 0 ? n : 0u);
            if (lane == kLong) n = longs;
            if (lane < kCounts) lcnt[lane] = n ? atomicAdd(q.scount + (size_t)b * kCounts + lane, n) : 0u;
        }
        __syncthreads();
        uint4* seg = q.seg + (size_t)b * q.sl.cap;
        for (uint32_t i = threadIdx.x; i < nc; i += kPartThreads) {
            const uint32_t f = found[i];
            if (!f) continue;
            const uint32_t hv = (uint32_t)(a[i] >> 32), len = (f >> 8) & 0xFFu, z = f & 0xFFu;
            const int cls = seg_class(len);
            // pair count: K + 1 for a source entry, 1 otherwise
            const uint4 d = make_uint4(pbase + start[(hv << log_parts) >> (32 - kLogSub)] + ((f >> 16) & 0xFFu), len,
                                       unhrow(hv), len + z * q.K);
            seg[q.sl.off[cls] + atomicAdd(lcnt + cls, 1u)] = d;
            if (cls > 0) seg[q.sl.off[kLong] + atomicAdd(lcnt + kLong, 1u)] = d;
        }
        __syncthreads();
    }
    // large sub-buckets: one warp each
    for (uint32_t g = warp; g < nbig; g += kPartThreads / 32) {
        const uint32_t s0 = start[big[g]], s1 = start[big[g] + 1];
        warp_sort_keys(aw + s0, s1 - s0);
        for (uint32_t h = s0; h < s1;) {
            // the segment that begins at h: its end, and its source entries
            const uint32_t hv = (uint32_t)(a[h] >> 32);
            uint32_t e = h, z = 0, in = 0xFFFFFFFFu;
            for (; in == 0xFFFFFFFFu && e < s1; e += 32) {
                const uint64_t key = e + lane < s1 ? a[e + lane] : 0ull;
                const bool same = e + lane < s1 && (uint32_t)(key >> 32) == hv;
                in = __ballot_sync(0xFFFFFFFFu, same);
                z += __popc(__ballot_sync(0xFFFFFFFFu, same && ((uint32_t)key & kSlotMask) == 0));
            }
            const uint32_t end = e - 32 + __popc(in), len = end - h;
            for (uint32_t i = h + lane; i < end; i += 32) {
                const uint32_t v = (uint32_t)a[i];
                q.slot_info[(v >> kSlotBits) * q.R + (v & kSlotMask)] = len == 1 ? kSingleBit : pbase + i;
            }
            list_segments(q, b, lane == 0, pbase + h, len, hv, z);
            h = end;
        }
    }
}

__global__ void __launch_bounds__(kPartThreads) k_group_parts(GroupParams q, int log_parts) {
    extern __shared__ uint64_t gkeys[];  // kPartCap keys, then the sub-buckets' counts and starts
    __shared__ uint32_t maps[2u << (kMapBits - 5)];  // hit once, hit twice
    uint32_t* const once = maps;
    uint32_t* const twice = maps + (1u << (kMapBits - 5));
    uint32_t* const cnt = reinterpret_cast<uint32_t*>(gkeys + kPartCap);  // keys per sub-bucket, then the next key's place
    uint32_t* const start = cnt + kPartSub;                               // [kPartSub + 1] sub-bucket starts
    __shared__ uint32_t lcnt[kCounts];        // segments per list, then the next one's place
    __shared__ uint32_t wtot[32];
    __shared__ uint16_t big[(kPartItems2 << kPartMaxLog) / kRankMax];
    __shared__ uint32_t nbig, pbase;
    constexpr int U = 8;  // record entries per thread loaded at once
    const uint32_t me = blockIdx.x, tid = threadIdx.x;
    const int b = blockIdx.y, lane = tid & 31, warp = tid >> 5;
    uint64_t base;
    uint32_t n;
    batch_range(q, b, &base, &n);
    const int32_t* rec = q.rec + base;
    const uint32_t s_base = (uint32_t)((int64_t)b * q.batch);
    for (uint32_t i = tid; i < 2u << (kMapBits - 5); i += kPartThreads) maps[i] = 0u;
    for (uint32_t i = tid; i < kPartSub; i += kPartThreads) cnt[i] = 0u;
    if (tid < kCounts) lcnt[tid] = 0u;
    if (tid == 0) nbig = 0;
    __syncthreads();
    // f(entry index, sample within the batch, slot, hrow) for each of the part's entries
    auto each = [&](auto&& f) {
        for (uint32_t r = tid; r < n; r += kPartThreads * U) {
            int32_t row[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const uint32_t i = r + k * kPartThreads;
                row[k] = i < n ? __ldg(rec + i) : 0;
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const uint32_t i = r + k * kPartThreads;
                const uint32_t smp = __umulhi(i, q.R_magic), slot = i - smp * q.R;
                const uint32_t hv = hrow((uint32_t)row[k] + (slot ? q.ctx_off : 0u));
                if (i < n && (log_parts == 0 || hv >> (32 - log_parts) == me)) f(i, smp, slot, hv);
            }
        }
    };
    each([&](uint32_t, uint32_t, uint32_t, uint32_t hv) {
        const uint32_t h = (hv << log_parts) >> (32 - kMapBits), bit = 1u << (h & 31u);
        if (atomicOr(&once[h >> 5], bit) & bit) atomicOr(&twice[h >> 5], bit);
        if (q.depmap) {
            const uint32_t db = hv >> (32 - kDepLog);
            atomicOr(q.depmap + (size_t)b * kDepWords + (db >> 5), 1u << (db & 31u));
        }
    });
    __syncthreads();
    each([&](uint32_t i, uint32_t, uint32_t, uint32_t hv) {
        const uint32_t h = (hv << log_parts) >> (32 - kMapBits);
        if (twice[h >> 5] >> (h & 31u) & 1u) atomicAdd(&cnt[(hv << log_parts) >> (32 - kLogSub)], 1u);
        else q.slot_info[base + i] = kSingleBit;
    });
    __syncthreads();
    // exclusive scan of the counts, four a thread
    uint4* const cnt4 = reinterpret_cast<uint4*>(cnt) + tid;
    const uint4 c4 = *cnt4;
    const uint32_t own = c4.x + c4.y + c4.z + c4.w;
    uint32_t incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) wtot[warp] = incl;
    __syncthreads();
    uint32_t wsum = lane < warp ? wtot[lane] : 0u;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) wsum += __shfl_xor_sync(0xFFFFFFFFu, wsum, o);
    uint4 st;
    st.x = wsum + incl - own;
    st.y = st.x + c4.x;
    st.z = st.y + c4.y;
    st.w = st.z + c4.z;
    *cnt4 = st;
    *(reinterpret_cast<uint4*>(start) + tid) = st;
    if (tid == kPartThreads - 1) {
        start[kPartSub] = wsum + incl;
        pbase = atomicAdd(q.pcount + b, wsum + incl);
    }
    // large sub-buckets (each has over kRankMax of the batch's items)
    if (c4.x > kRankMax) big[atomicAdd(&nbig, 1u)] = (uint16_t)(4 * tid);
    if (c4.y > kRankMax) big[atomicAdd(&nbig, 1u)] = (uint16_t)(4 * tid + 1);
    if (c4.z > kRankMax) big[atomicAdd(&nbig, 1u)] = (uint16_t)(4 * tid + 2);
    if (c4.w > kRankMax) big[atomicAdd(&nbig, 1u)] = (uint16_t)(4 * tid + 3);
    __syncthreads();
    const uint32_t nc = start[kPartSub];
    const bool fits = nc <= kPartCap;
    uint64_t* far = q.bucketed + base + pbase;  // a part too large for shared memory (a very skewed draw)
    each([&](uint32_t, uint32_t smp, uint32_t slot, uint32_t hv) {
        const uint32_t h = (hv << log_parts) >> (32 - kMapBits);
        if (twice[h >> 5] >> (h & 31u) & 1u) {
            const uint32_t at = atomicAdd(&cnt[(hv << log_parts) >> (32 - kLogSub)], 1u);
            const uint64_t key = ((uint64_t)hv << 32) | ((s_base + smp) << kSlotBits | slot);
            if (fits) gkeys[at] = key;
            else far[at] = key;
        }
    });
    __syncthreads();
    if (fits) group_segments(q, gkeys, gkeys, nc, start, log_parts, pbase, b, big, nbig, maps, lcnt);
    else group_segments(q, far, far, nc, start, log_parts, pbase, b, big, nbig, maps, lcnt);
}

// ---------------------------------------------------------------------------
// Workspace.
// ---------------------------------------------------------------------------
struct Buf {
    void* p = nullptr;
    size_t cap = 0;
    cudaError_t ensure(size_t bytes, DeviceScratch* kept) {
        if (bytes <= cap) return cudaSuccess;
        if (p) cudaFree(p);
        p = nullptr;
        cap = 0;
        cudaError_t e = device_alloc(&p, bytes, kept);
        if (e == cudaSuccess) cap = bytes;
        return e;
    }
    ~Buf() {
        if (p) cudaFree(p);
    }
};

// A data phase captured as a CUDA graph, and what it was captured for: the
// parameters, the warps per block and the kernels (the launcher of one row
// width and table type: tables of another type can sit at the same addresses).
// A capture takes about 2.2 us a launch more than launching, a replay saves
// 0.3 us of each: a phase that recurs from call to call is captured when it
// has been launched kCaptureAfter times in a row, so that no sequence of calls
// pays more for captures than about what it has to gain (captured at the first
// repetition, two calls of one kind after two of another took 19% longer than
// without: 12.4 against 10.4 ms for four of 100,000 samples at B = 256).
constexpr int kCaptureAfter = 8;

struct CapturedPhase {
    using Fn = cudaError_t (*)(const DataParams&, int, cudaStream_t);
    cudaGraphExec_t exec = nullptr;  // null: `key` was met, not captured yet
    DataParams key{};
    int wpb = -1;
    Fn fn = nullptr;
    int met = 0;  // direct launches of `key` in a row
    bool is(const DataParams& k, int w, Fn f) const { return fn == f && wpb == w && memcmp(&k, &key, sizeof k) == 0; }
};

// Per-chunk outputs of the pre-pass, read by the data phase.  Two sets: the
// pre-pass of chunk c+1 (on its own low-priority stream) fills one while the
// data phase of chunk c reads the other.
struct ChunkSet {
    Buf rec, slot_info, depmap, seg, scount, bpar;
    // captured data phases of this set: of a full chunk, and of the shorter
    // one that ends a call
    CapturedPhase captured[2];
    cudaEvent_t prep_done = nullptr;  // pre-pass of the set's current chunk finished
    cudaEvent_t data_done = nullptr;  // data phase of the set's previous chunk finished
    bool data_pending = false;
};

struct TrainWorkspace {
    Buf items0, items1, gcnt, boff, pcount, counters, slab, gbar;
    ChunkSet set[2];
    cudaStream_t prep = nullptr;    // pre-pass stream
    cudaStream_t cap = nullptr;     // stream the data-phase graphs are captured on
    bool graph_failed = false;      // a capture failed: direct launches from then on
    cudaEvent_t start = nullptr;    // caller-stream work before the call
    std::vector<cudaEvent_t> events;  // timing events
    cudaError_t event(size_t i, cudaEvent_t* out) {
        while (events.size() <= i) {
            cudaEvent_t e;
            cudaError_t r = cudaEventCreate(&e);
            if (r != cudaSuccess) return r;
            events.push_back(e);
        }
        *out = events[i];
        return cudaSuccess;
    }
    cudaError_t init(int device) {
        if (prep) return cudaSuccess;
        int lo = 0, hi = 0;
        cudaError_t e = cudaDeviceGetStreamPriorityRange(&lo, &hi);
        if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&prep, cudaStreamNonBlocking, lo);
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
        for (auto& cs : set) {
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&cs.prep_done, cudaEventDisableTiming);
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&cs.data_done, cudaEventDisableTiming);
        }
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&start, cudaEventDisableTiming);
        (void)device;
        return e;
    }
    ~TrainWorkspace() {
        if (prep) {
            cudaStreamSynchronize(prep);
            cudaStreamDestroy(prep);
        }
        if (cap) cudaStreamDestroy(cap);
        for (auto& cs : set) {
            if (cs.prep_done) cudaEventDestroy(cs.prep_done);
            if (cs.data_done) cudaEventDestroy(cs.data_done);
            for (auto& g : cs.captured)
                if (g.exec) cudaGraphExecDestroy(g.exec);
        }
        if (start) cudaEventDestroy(start);
        for (auto e : events) cudaEventDestroy(e);
    }
};

TrainWorkspace* workspace_create() { return new TrainWorkspace(); }
void workspace_destroy(TrainWorkspace* ws) { delete ws; }

static uint32_t bits_for(uint64_t v) {  // bits to hold values 0..v-1
    uint32_t b = 1;
    while ((1ull << b) < v) ++b;
    return b;
}

// Runs f once per device (function attributes are per device); thread-safe.
template <typename F>
static void once_per_device(std::atomic<uint64_t>& done, F f) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    const uint64_t bit = 1ull << (dev & 63);
    if (done.load(std::memory_order_acquire) & bit) return;
    f();
    done.fetch_or(bit, std::memory_order_acq_rel);
}

// Warps of a staged gather block (at most kGatherWarps, fewer when the stages
// exceed the shared memory) and its shared memory.
template <int D, int DT>
static int staged_warps(int K, int requested, size_t* smem_out) {
    // staging: K+1 context rows per lane group
    const size_t per_warp = (size_t)(K + 1) * Geom<D, DT>::GPW * D * (DT == LINE_DTYPE_F32 ? 4 : 2);
    // (2 warps a block: 3.72 ms for 2^19 samples at d = 256, K = 10, with 4
    // 3.99; narrower rows within 1%)
    const int wpb = requested > 0 ? std::min(requested, kGatherWarps) : 2;
    const int fit = std::max(1, std::min(wpb, (int)(kMaxSmem / per_warp)));
    *smem_out = (size_t)fit * per_warp;
    return fit;
}

template <int D, int DT>
static cudaError_t launch_data_batched(const DataParams& p, int warps_per_block, cudaStream_t s) {
    using G = Geom<D, DT>;
    // 4 warps per block: at 64 registers a 4096-sample batch is one wave.
    // Rows of up to 128 values and K <= 7: the context rows in registers, in
    // the smallest body that holds them (K + 1 <= 2, 4, 6 or 8)
    size_t smem = 0;
    int wpb = warps_per_block > 0 ? std::min(warps_per_block, kGatherWarps) : kGatherWarps;
    void (*gather)(DataParams, int) = nullptr;
    if constexpr (G::E <= 4) {
        if (p.K < 8)
            gather = p.K < 2 ? k_gather<D, DT, 2> : p.K < 4 ? k_gather<D, DT, 4> : p.K < 6 ? k_gather<D, DT, 6> : k_gather<D, DT, 8>;
    }
    if (!gather) {
        gather = k_gather<D, DT, 0>;
        wpb = staged_warps<D, DT>(p.K, warps_per_block, &smem);
        static std::atomic<uint64_t> attr_set{0};
        once_per_device(attr_set, [] {
            cudaFuncSetAttribute(k_gather<D, DT, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
        });
    }
    const int64_t per_block = (int64_t)wpb * G::GPW;
    const int aw = p.apply_warps == kApplyWarpsAlone && D <= 128 ? kApplyWarpsAlone : kApplyWarpsShared;
    // blocks for the short segments, at most (R-MAT 20 has about 3,000 of them
    // a batch).  2^22 samples, one order BF16 with 152, 228 and 304 blocks of
    // 16 warps: 7.36, 6.55 and 6.50 ms; both orders FP32 with 152, 304, 456 and
    // 608 of 8: 12.44, 11.41, 11.24 and 11.46; d = 256 with 304 of 16: 5.27 for
    // 2^19, with 608 of 8 (which leave registers for the gather's): 4.83
    const int64_t short_blocks = aw == kApplyWarpsAlone ? 304 : D <= 128 ? 456 : 608;
    const int64_t apply_per_block = (int64_t)aw * G::GPW;
    cudaError_t e = cudaSuccess;
    for (int b = 0; b < p.n_batches && e == cudaSuccess; ++b) {
        const int64_t nb = std::min<int64_t>(p.batch, p.chunk_samples - (int64_t)b * p.batch);
        const unsigned g1 = (unsigned)((nb + per_block - 1) / per_block);
        // the chunk's first gather follows the pre-pass with a full dependency;
        // later launches overlap their start with the previous kernel's tail
        e = launch_pdl(gather, g1, wpb * 32, smem, s, b > 0, p, b);
        if (e != cudaSuccess) break;
        // a shared segment has two or more of the batch's nb * (K+2) entries
        const int64_t max_m = nb * (p.K + 2) / 2 + 1;
        const unsigned g2 = 1024 / aw + (unsigned)std::min<int64_t>((max_m + apply_per_block - 1) / apply_per_block, short_blocks);
        if (aw == kApplyWarpsAlone) e = launch_pdl(k_apply<D, DT, kApplyWarpsAlone>, g2, kApplyWarpsAlone * 32, 0, s, true, p, b);
        else e = launch_pdl(k_apply<D, DT, kApplyWarpsShared>, g2, kApplyWarpsShared * 32, 0, s, true, p, b);
    }
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

template <int D, int DT>
static cudaError_t launch_data_persistent(const DataParams& p, int warps_per_block, cudaStream_t s) {
    using G = Geom<D, DT>;
    int dev = 0, sms = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    int W = warps_per_block > 0 ? std::min(warps_per_block, kPersistMaxWarps) : kPersistDefaultWarps;
    // two row slots per warp when a warp has two or more units of a batch
    auto slots_for = [&](int w) {
        const int64_t units = (p.batch + G::GPW - 1) / G::GPW;
        return units > (int64_t)sms * w ? 2 : 1;
    };
    size_t smem = persist_smem_bytes(D, DT, p.K, W, slots_for(W), G::GPW);
    while (W > 1 && smem > (size_t)optin) {
        --W;
        smem = persist_smem_bytes(D, DT, p.K, W, slots_for(W), G::GPW);
    }
    if (smem > (size_t)optin) return cudaErrorInvalidConfiguration;
    if ((e = cudaFuncSetAttribute(k_persistent<D, DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
        cudaSuccess)
        return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_persistent<D, DT>, W * 32, smem)) != cudaSuccess)
        return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    DataParams pc = p;
    pc.slots = slots_for(W);
    if ((e = cudaMemsetAsync(p.gbar, 0, 2 * sizeof(uint32_t), s)) != cudaSuccess) return e;
    void* args[] = {&pc};
    return cudaLaunchCooperativeKernel((const void*)k_persistent<D, DT>, dim3((unsigned)sms), dim3((unsigned)(W * 32)),
                                       args, smem, s);
}

using LaunchFn = cudaError_t (*)(const DataParams&, int, cudaStream_t);

static LaunchFn pick_launcher(int dim, int dtype, bool persistent) {
#define LINE_PICK(DD)                                                                                   \
    if (dim == DD) {                                                                                    \
        if (persistent)                                                                                 \
            return dtype == LINE_DTYPE_F32 ? launch_data_persistent<DD, LINE_DTYPE_F32>                 \
                                           : launch_data_persistent<DD, LINE_DTYPE_BF16>;               \
        return dtype == LINE_DTYPE_F32 ? launch_data_batched<DD, LINE_DTYPE_F32>                        \
                                       : launch_data_batched<DD, LINE_DTYPE_BF16>;                      \
    }
    LINE_PICK(16)
    LINE_PICK(32)
    LINE_PICK(64)
    LINE_PICK(128)
    LINE_PICK(256)
#undef LINE_PICK
    return nullptr;
}

cudaError_t train_run(const TrainArgs& a, TrainWorkspace* ws, uint32_t* status, TrainTimes* times, cudaStream_t s,
                      std::string* err) {
    const int R = a.K + 2;
    const uint64_t n_samples = a.t_end - a.t_begin;
    if (n_samples == 0) return cudaSuccess;
    const uint64_t rows_space = a.order == 2 ? 2ull * (uint64_t)a.n_nodes : (uint64_t)a.n_nodes;
    const uint32_t row_bits = bits_for(rows_space);
    if (row_bits > 31) {
        *err = "too many nodes for 32-bit row ids";
        return cudaErrorInvalidValue;
    }
    // batches per chunk: about 2^18 samples (2^20 for walk pairs in the
    // Hogwild schedule, whose faster update launch would otherwise wait for
    // the next chunk's walks: a walk's steps are sequential, so a chunk's
    // walks take about the same time whatever their number), limited by
    // 31-bit positions and by the chunk-sample field of item values
    const bool long_chunks = a.mode == LINE_MODE_HOGWILD && a.walk_len > 0;
    int64_t nb = a.chunk_batches > 0 ? a.chunk_batches
                                     : std::max<int64_t>(1, (int64_t(1) << (long_chunks ? 20 : 18)) / a.batch);
    while (nb > 1 && ((uint64_t)nb * (uint64_t)a.batch * (uint64_t)R >= (1ull << 31) ||
                      (uint64_t)nb * (uint64_t)a.batch > (1ull << (32 - kSlotBits))))
        nb >>= 1;
    const uint64_t total_batches = (n_samples + a.batch - 1) / a.batch;
    nb = (int64_t)std::min<uint64_t>((uint64_t)nb, total_batches);
    const int64_t max_chunk = nb * a.batch;
    const int64_t max_items = max_chunk * R;
    const uint32_t parts = (uint32_t)((a.batch * R + kPartItems - 1) / kPartItems);
    // batches of up to 16 parts of 16,384 items are grouped part by part in
    // shared memory (every part scans the whole batch); larger ones are
    // bucketed through global memory first
    int log_parts = 0;
    while (a.batch * R > ((int64_t)kPartItems2 << log_parts)) ++log_parts;
    const bool direct = log_parts <= kPartMaxLog;
    // the persistent schedule needs all its CTAs resident at once, which a
    // second cooperative launch on the other order's stream could prevent:
    // concurrent orders run the batched schedule
    const bool persistent = a.mode == LINE_MODE_PERSISTENT && !a.concurrent;
    const bool hogwild = a.mode == LINE_MODE_HOGWILD;  // records only: no grouping, slab or apply
    SegLayout sl;
    sl.set(a.batch * R);

    cudaError_t e;
    auto ensure = [&](Buf& b, size_t bytes) -> bool {
        if ((e = b.ensure(bytes, a.kept)) != cudaSuccess) {
            *err = "device allocation failed (training scratch)";
            return false;
        }
        return true;
    };
    int device = 0;
    if ((e = cudaGetDevice(&device)) != cudaSuccess) return e;
    if ((e = ws->init(device)) != cudaSuccess) return e;
    // every scratch buffer and its size for this call
    auto each = [&](auto&& f) -> bool {
        if (hogwild) {
            for (auto& cs : ws->set)
                if (!f(cs.rec, sizeof(int32_t) * max_items)) return false;
            return true;
        }
        if (!f(ws->items1, sizeof(uint64_t) * max_items) || !f(ws->counters, 256) ||
            !f(ws->pcount, sizeof(uint32_t) * (nb + 1)) ||
            !f(ws->slab, sizeof(float) * (size_t)std::min<int64_t>(max_items, a.batch * R) * a.dim))
            return false;
        if (!direct && (!f(ws->items0, sizeof(uint64_t) * max_items) ||
                        !f(ws->gcnt, sizeof(uint32_t) * (size_t)nb * parts * kBuckets) ||
                        !f(ws->boff, sizeof(uint32_t) * (size_t)nb * (kBuckets + 1))))
            return false;
        for (auto& cs : ws->set) {
            if (!f(cs.rec, sizeof(int32_t) * max_items) || !f(cs.bpar, sizeof(BatchParams) * (nb + 1)) ||
                !f(cs.slot_info, sizeof(uint32_t) * max_items) || !f(cs.seg, sizeof(uint4) * (size_t)nb * sl.cap) ||
                !f(cs.scount, sizeof(uint32_t) * (size_t)nb * kCounts))
                return false;
            if (persistent && !f(cs.depmap, sizeof(uint32_t) * (size_t)nb * kDepWords)) return false;
        }
        return true;
    };
    // Buffers still used by an earlier call's data phase are reallocated
    // only after that phase is done; when nothing grows, consecutive calls on
    // the stream pipeline (the chunk sets' events order the reuse).
    bool grow = false;
    each([&](Buf& b, size_t bytes) {
        grow = grow || b.cap < bytes;
        return true;
    });
    if (grow) {
        if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
        if (ws->prep && (e = cudaStreamSynchronize(ws->prep)) != cudaSuccess) return e;
        for (auto& cs : ws->set) cs.data_pending = false;
        if (!each(ensure)) return e;
    }
    if (persistent && !ensure(ws->gbar, 256)) return e;
    LaunchFn data = pick_launcher(a.dim, a.dtype, persistent);
    if (!data) {
        *err = "unsupported dim";
        return cudaErrorInvalidValue;
    }
    const size_t sort_smem = (size_t)kSortBucketsPerCta * 2 * kWarpSortCap * sizeof(uint64_t);
    const size_t group_smem = (size_t)kPartCap * sizeof(uint64_t) + sizeof(uint32_t) * (2 * (size_t)kPartSub + 4);
    if ((e = cudaFuncSetAttribute(k_bucket_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sort_smem)) !=
            cudaSuccess ||
        (e = cudaFuncSetAttribute(k_group_parts, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)group_smem)) !=
            cudaSuccess)
        return e;
    cudaStream_t ps = ws->prep;
    // the pre-pass reads the graph and alias tables made on the caller's stream
    if ((e = cudaEventRecord(ws->start, s)) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(ps, ws->start, 0)) != cudaSuccess) return e;

    PrepassParams pp{};
    pp.src = a.src;
    pp.dst = a.dst;
    pp.edge_tab = a.edge_tab;
    pp.neg_tab = a.neg_tab;
    pp.n_arcs = a.n_arcs;
    pp.n_nodes = a.n_nodes;
    pp.seed = a.seed;
    pp.batch = a.batch;
    pp.K = a.K;
    pp.order = a.order;
    pp.walk = a.walk_len > 0;
    pp.lr0 = (float)a.lr0;
    pp.lr_floor = (float)a.lr_floor;
    pp.lr_schedule = a.lr_schedule;
    pp.lr_total = a.lr_total;
    pp.pcount = (uint32_t*)ws->pcount.p;

    WalkParams wp{};
    if (a.walk_len > 0) {
        wp.src = a.src;
        wp.dst = a.dst;
        wp.edge_tab = a.edge_tab;
        wp.n_arcs = a.n_arcs;
        wp.row_ptr = a.row_ptr;
        wp.cw = a.cw;
        wp.seed = a.seed;
        wp.L = a.walk_len;
        wp.W = a.window;
        wp.P = (uint64_t)a.walk_len * a.window - (uint64_t)a.window * (a.window - 1) / 2;
        wp.reuse = (uint32_t)a.walk_reuse;
        wp.R = (uint64_t)R;
    }

    GroupParams gq{};
    gq.batch = a.batch;
    gq.R = (uint32_t)R;
    gq.K = (uint32_t)a.K;
    gq.parts = parts;
    gq.R_magic = (uint32_t)(((uint64_t)1 << 32) / (uint32_t)R) + 1u;
    gq.ctx_off = a.order == 2 ? (uint32_t)a.n_nodes : 0u;
    gq.bucketed = (uint64_t*)ws->items1.p;
    gq.tmp = (uint64_t*)ws->items0.p;
    gq.pcount = (uint32_t*)ws->pcount.p;
    gq.gcnt = (uint32_t*)ws->gcnt.p;
    gq.boff = (uint32_t*)ws->boff.p;
    gq.sl = sl;

    uint32_t* abort_word = (uint32_t*)ws->counters.p + 16;

    DataParams dp{};
    dp.U = a.U;
    dp.C = a.order == 2 ? a.C : a.U;
    dp.order = a.order;
    dp.K = a.K;
    dp.n_nodes = a.n_nodes;
    dp.row_bits = row_bits;
    dp.sl = sl;
    dp.slab = (float*)ws->slab.p;
    dp.batch = a.batch;
    dp.lambda = (float)a.lambda;
    dp.alpha_neg = (float)a.alpha_neg;
    dp.status = status;
    dp.gbar = (uint32_t*)ws->gbar.p;
    dp.spin_limit = a.spin_limit;
    dp.abort_word = abort_word;
    dp.apply_warps = a.concurrent ? kApplyWarpsShared : kApplyWarpsAlone;

    struct ChunkRec {
        size_t ev;  // events ev, ev+1 (pre-pass stream), ev+2, ev+3 (data stream)
    };
    std::vector<ChunkRec> chunk_log;
    size_t n_ev = 0;
    cudaEvent_t ev = nullptr;
    int c = 0;
    for (uint64_t t = a.t_begin; t < a.t_end; t += (uint64_t)max_chunk, ++c) {
        ChunkSet& cset = ws->set[c & 1];
        const int64_t cs = (int64_t)std::min<uint64_t>((uint64_t)max_chunk, a.t_end - t);
        const int cb = (int)((cs + a.batch - 1) / a.batch);
        const int64_t n_items = cs * R;
        int launches = 0;
        // ---- pre-pass of chunk c on the pre-pass stream, into set c % 2,
        // once the data phase of chunk c-2 (the set's last reader) is done
        if (cset.data_pending && (e = cudaStreamWaitEvent(ps, cset.data_done, 0)) != cudaSuccess) return e;
        if (a.timing) {
            if ((e = ws->event(n_ev, &ev)) != cudaSuccess) return e;
            cudaEventRecord(ev, ps);
        }
        pp.t_chunk = t;
        pp.chunk_samples = cs;
        pp.rec = (int32_t*)cset.rec.p;
        if (!hogwild) {
            pp.n_batches = cb;
            pp.bpar = (BatchParams*)cset.bpar.p;
            pp.scount = (uint32_t*)cset.scount.p;
        }
        {
            const int64_t work = cs * (a.K + 1);
            const unsigned g = (unsigned)std::min<int64_t>((work + 255) / 256, 152 * 64);
            k_chunk_draws<<<g, 256, 0, ps>>>(pp);
            if (a.walk_len > 0) {
                wp.t0 = t;
                wp.count = cs;
                wp.rec = (int32_t*)cset.rec.p;
                if ((e = walk_pairs(wp, ps)) != cudaSuccess) return e;
                ++launches;
            }
        }
        if (!hogwild) {
            gq.n_batches = cb;
            gq.chunk_samples = cs;
            gq.rec = (const int32_t*)cset.rec.p;
            gq.slot_info = (uint32_t*)cset.slot_info.p;
            gq.seg = (uint4*)cset.seg.p;
            gq.scount = (uint32_t*)cset.scount.p;
            gq.depmap = persistent ? (uint32_t*)cset.depmap.p : nullptr;
            if (persistent &&
                (e = cudaMemsetAsync(cset.depmap.p, 0, sizeof(uint32_t) * (size_t)cb * kDepWords, ps)) != cudaSuccess)
                return e;
            if (direct) {
                k_group_parts<<<dim3(1u << log_parts, cb), kPartThreads, group_smem, ps>>>(gq, log_parts);
                launches += 2;
            } else {
                k_bucket_count<<<dim3(parts, cb), kBucketThreads, 0, ps>>>(gq);
                k_bucket_scatter<<<dim3(parts, cb), kBucketThreads, 0, ps>>>(gq);
                k_bucket_sort<<<dim3(kBuckets / kSortBucketsPerCta, cb), kSortThreads, sort_smem, ps>>>(gq);
                launches += 4;
            }
        } else {
            launches += 1;  // the draws alone
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (a.timing) {
            if ((e = ws->event(n_ev + 1, &ev)) != cudaSuccess) return e;
            cudaEventRecord(ev, ps);
        }
        if ((e = cudaEventRecord(cset.prep_done, ps)) != cudaSuccess) return e;
        // ---- data phase of chunk c on the caller's stream
        if ((e = cudaStreamWaitEvent(s, cset.prep_done, 0)) != cudaSuccess) return e;
        if (a.timing) {
            if ((e = ws->event(n_ev + 2, &ev)) != cudaSuccess) return e;
            cudaEventRecord(ev, s);
        }
        if (hogwild) {
            HogwildParams hp{};
            hp.U = a.U;
            hp.C = a.C;
            hp.order = a.order;
            hp.K = a.K;
            hp.n_nodes = a.n_nodes;
            hp.rec = (const int32_t*)cset.rec.p;
            hp.chunk_samples = cs;
            hp.t_chunk = t;
            hp.batch = a.batch;
            hp.lr0 = (float)a.lr0;
            hp.lr_floor = (float)a.lr_floor;
            hp.lr_schedule = a.lr_schedule;
            hp.lr_total = a.lr_total;
            hp.lambda = (float)a.lambda;
            hp.alpha_neg = (float)a.alpha_neg;
            hp.seed = a.seed;
            hp.status = status;
            if ((e = hogwild_chunk(hp, a.dim, a.dtype, a.hogwild_workers, s)) != cudaSuccess) return e;
        } else {
            dp.rec = (const int32_t*)cset.rec.p;
            dp.slot_info = (const uint32_t*)cset.slot_info.p;
            dp.seg = (const uint4*)cset.seg.p;
            dp.scount = (const uint32_t*)cset.scount.p;
            dp.bpar = (const BatchParams*)cset.bpar.p;
            dp.depmap = (const uint32_t*)cset.depmap.p;
            dp.chunk_samples = cs;
            dp.n_batches = cb;
            if (persistent && (e = cudaMemsetAsync(abort_word, 0, sizeof(uint32_t), s)) != cudaSuccess) return e;
            // A chunk's launches are replayed from a captured graph (what differs
            // from chunk to chunk is in the set's buffers) when it is a full chunk
            // after the first of its call, or when the set's last chunks of its
            // kind, full or not, were the same: a call of few chunks that is
            // repeated.  A launch costs 2.3 us of host time, two a batch: with
            // both orders at B = 256 the launches, not the GPU, set the pace
            // (7.7 us a batch; 4.6 replayed).
            CapturedPhase& cap = cset.captured[cs == max_chunk ? 0 : 1];
            const bool known = cap.is(dp, a.warps_per_block, data);
            if (!persistent && a.graph && !ws->graph_failed &&
                ((known && (cap.exec || cap.met >= kCaptureAfter)) || (cs == max_chunk && c > 0))) {
                if (!known || !cap.exec) {
                    if (cap.exec) cudaGraphExecDestroy(cap.exec);
                    cap = CapturedPhase{};
                    cudaGraph_t g = nullptr;
                    cudaError_t ce = cudaStreamBeginCapture(ws->cap, cudaStreamCaptureModeThreadLocal);
                    if (ce == cudaSuccess) {
                        const cudaError_t le = data(dp, a.warps_per_block, ws->cap);
                        ce = cudaStreamEndCapture(ws->cap, &g);
                        if (ce == cudaSuccess) ce = le;
                    }
                    if (ce == cudaSuccess) ce = cudaGraphInstantiate(&cap.exec, g, 0);
                    if (g) cudaGraphDestroy(g);
                    if (ce != cudaSuccess) {
                        cudaGetLastError();
                        cap.exec = nullptr;
                        ws->graph_failed = true;
                    } else {
                        cap.key = dp;
                        cap.wpb = a.warps_per_block;
                        cap.fn = data;
                    }
                }
                e = cap.exec ? cudaGraphLaunch(cap.exec, s) : data(dp, a.warps_per_block, s);
                if (e != cudaSuccess) return e;
            } else {
                if (!persistent) {
                    if (!known) {
                        if (cap.exec) cudaGraphExecDestroy(cap.exec);
                        cap = CapturedPhase{nullptr, dp, a.warps_per_block, data};
                    }
                    ++cap.met;
                }
                if ((e = data(dp, a.warps_per_block, s)) != cudaSuccess) return e;
            }
        }
        if (a.timing) {
            if ((e = ws->event(n_ev + 3, &ev)) != cudaSuccess) return e;
            cudaEventRecord(ev, s);
            chunk_log.push_back({n_ev});
            n_ev += 4;
        }
        if ((e = cudaEventRecord(cset.data_done, s)) != cudaSuccess) return e;
        cset.data_pending = true;
        // launches counted whether or not they are timed (a graph replay
        // counts the kernels it holds)
        times->prepass_launches += launches;
        times->update_launches += (persistent || hogwild) ? 1 : 2 * (int64_t)cb;
        times->update_samples += (uint64_t)cs;
    }
    // the pre-pass stream's work is all ordered before the last data phase
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (a.timing && n_ev) {
        if ((e = cudaEventSynchronize(ws->events[n_ev - 1])) != cudaSuccess) return e;
        for (const ChunkRec& r : chunk_log) {
            float ms1 = 0, ms2 = 0;
            cudaEventElapsedTime(&ms1, ws->events[r.ev], ws->events[r.ev + 1]);
            cudaEventElapsedTime(&ms2, ws->events[r.ev + 2], ws->events[r.ev + 3]);
            times->prepass_ms += ms1;
            times->update_ms += ms2;
        }
    }
    return cudaSuccess;
}

}  // namespace line
