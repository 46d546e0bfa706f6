// Pieces shared by the kernels that keep their chunk partial sums in tensor memory
// (layer_resident.cu: one layer per launch; model_kernel.cu: many layers per launch).
#pragma once
#include "ptx.cuh"

#include <cuda_runtime.h>
#include <stdint.h>

namespace chunkkv {

constexpr int kRUmmaN = 128;                 // UMMA N (a multiple of 16): a tile of 120 keys leaves the last 8 columns unread
constexpr int kRPanel = 60;                  // keys per epilogue panel (half a tile)
constexpr int kRMaxStages = 14;
constexpr int kRPartCol0 = 256;              // tensor-memory column of the first chunk partial sum
constexpr int kRPartCols = 256;
constexpr int kRQTileBytes = 128 * 128;

// Keys per epilogue panel (half a tile) for a chunk size: a multiple of it, so that no chunk straddles panels.
__host__ __device__ constexpr int panel_keys(int c) { return (c == 8 || c == 16 || c == 32) ? 64 : kRPanel; }

// One accumulator tile: the products of 64 or 128 dims, four of 16 dims per ring stage (k-steps advance the start address by 32
// bytes). The descriptors come ready made, so that the issuing thread only adds constants between two products.
__device__ __forceinline__ void issue_products(uint32_t d_addr, uint64_t q_desc, uint64_t k_desc0, uint64_t k_desc1, bool both, uint32_t idesc) {
#pragma unroll
    for (int k4 = 0; k4 < 4; ++k4) umma_bf16(d_addr, q_desc + 2u * k4, k_desc0 + 2u * k4, idesc, k4 > 0 ? 1u : 0u);
    if (both) {
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4) umma_bf16(d_addr, q_desc + (kRQTileBytes >> 4) + 2u * k4, k_desc1 + 2u * k4, idesc, 1u);
    }
}

// A panel's chunk partial sums to and from consecutive tensor-memory columns.
template <int N>
__device__ __forceinline__ void part_store(uint32_t taddr, const float (&p)[N]) {
    constexpr int X4 = N / 4 * 4, X2 = X4 + (N & 2);
#pragma unroll
    for (int o = 0; o < X4; o += 4) tmem_st_x4(taddr + o, &p[o]);
    if constexpr ((N & 2) != 0) tmem_st_x2(taddr + X4, &p[X4]);
    if constexpr ((N & 1) != 0) tmem_st_x1(taddr + X2, &p[X2]);
}
template <int N>
__device__ __forceinline__ void part_load(uint32_t taddr, float* p) {
    constexpr int X4 = N / 4 * 4, X2 = X4 + (N & 2);
#pragma unroll
    for (int o = 0; o < X4; o += 4) tmem_ld_x4(taddr + o, p + o);
    if constexpr ((N & 2) != 0) tmem_ld_x2(taddr + X4, p + X4);
    if constexpr ((N & 1) != 0) tmem_ld_x1(taddr + X2, p + X2);
}

// Sum of 32 values per lane over the 32 lanes of a warp, transposed: lane j returns the sum over
// all lanes of their v[j]. 31 shuffles instead of 32 x 5 (each step halves the values a lane holds).
__device__ __forceinline__ float warp_transpose_reduce(float (&v)[32], int lane) {
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < off; ++i) {
            const float send = up ? v[i] : v[i + off];
            const float keep = up ? v[i + off] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    return v[0];
}

// Named barrier for a subset of the CTA's warps (id 1..15; id 0 is __syncthreads).
__device__ __forceinline__ void named_barrier(int id, int nthreads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// The same, returning to every participating thread whether any of them passed a true predicate.
__device__ __forceinline__ bool named_barrier_or(int id, int nthreads, bool pred) {
    uint32_t out;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %3, 0;\n\t"
        "barrier.cta.red.or.pred q, %1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(out)
        : "r"(id), "r"(nthreads), "r"(static_cast<uint32_t>(pred))
        : "memory");
    return out != 0;
}

// Merge (max, sum-of-exp2) pairs: (M, S) <- (M, S) (+) (m, s), all in the log2 domain, -inf: nothing yet. One exponential: the larger
// maximum's sum keeps its place. (Maxima rounded to whole numbers would need none, but the largest elements, whose exponential is
// exactly 1 as it is, then carry its error: 62261 tokens 4.1e-7 instead of 2.9e-7 of the token scores against 64 bits.)
__device__ __forceinline__ void merge_ml(float& M, float& S, float m, float s) {
    const float nm = fmaxf(M, m), e = M == m ? 1.f : ex2_approx(-fabsf(M - m));
    S = m > M ? fmaf(S, e, s) : fmaf(s, e, S);
    M = nm;
}

// The same for N records at a time: the largest maximum first, then each record's sum with one factor.
template <int N>
__device__ __forceinline__ void merge_records(float& M, float& S, const float (&m)[N], const float (&l)[N]) {
    float bm = M;
#pragma unroll
    for (int u = 0; u < N; ++u) bm = fmaxf(bm, m[u]);
    float acc = S * ex2_below(M, bm);
#pragma unroll
    for (int u = 0; u < N; ++u) acc += l[u] * ex2_below(m[u], bm);
    M = bm;
    S = acc;
}

// Up to KF records of a row (one every `step`, from `src`) in one round trip, as often as it takes until all of them carry this
// launch's tag; merged into (M, S), all at once or one after the other. False: given up.
template <int KF, bool IN_TURN>
__device__ __forceinline__ bool take_records(const ulonglong2* src, size_t step, int n, uint32_t tag, float& M, float& S, volatile int* abort_flag) {
    ulonglong2 r[KF];
    unsigned missing = (1u << n) - 1u;
    long long t0 = 0;
    for (uint32_t it = 1;; ++it) {
#pragma unroll
        for (int u = 0; u < KF; ++u)
            if (missing >> u & 1u) r[u] = ld_tagged2(src + u * step);
#pragma unroll
        for (int u = 0; u < KF; ++u)
            if ((missing >> u & 1u) && tagged_is(r[u].x, tag) && tagged_is(r[u].y, tag)) missing &= ~(1u << u);
        if (missing == 0u) break;
        if ((it & 63u) == 0u) {
            if (t0 == 0) t0 = clock64();
            if (*abort_flag) return false;
            if (clock64() - t0 > kWaitLimitClocks) { *abort_flag = 1; return false; }
        }
    }
    float m[KF], l[KF];
#pragma unroll
    for (int u = 0; u < KF; ++u) {
        m[u] = u < n ? tagged_value(r[u].x) : __int_as_float(0xff800000);
        l[u] = u < n ? tagged_value(r[u].y) : 0.f;
    }
    if constexpr (IN_TURN) {
#pragma unroll
        for (int u = 0; u < KF; ++u) merge_ml(M, S, m[u], l[u]);
    } else {
        merge_records(M, S, m, l);
    }
    return true;
}

// Hand-overs of the launches that have the GPU to themselves carry their data, which leaves out the release, the
// counter and the read behind it: two round trips of the L2 for each of the two (2048 tokens, 2 heads 11.84 -> 11.06 us, 8192 16.3 -> 15.4,
// 32768 29.2 -> 28.7, 9 CTAs a head 15.6 -> 14.6, 74 22.26 -> 21.31). The tag is the launch's number, so nothing
// has to be cleared. Launches that share the GPU with others of their kind (lanes) keep the counters and their own scratch.
// Launches on one scratch buffer are ordered, so one set of words each is enough; whose words a call gets: api.cu, take_exchange.
constexpr int kXScores = 65536;        // chunk scores of all scoring heads that fit (more: the second hand-over by counters)
struct Exchange {
    uint32_t last_tag;                 // of the launches so far
    uint32_t started;                  // CTAs of this launch that have taken its tag
    alignas(128) ulonglong2 record[kExchangeCtas * 2 * 128];       // [CTA, query tile][row]: maximum, sum
    ulonglong2 score[kXScores / 2];    // [scoring head][score_row / 2]
    __device__ void clear() {
        for (ulonglong2& x : record) x = make_ulonglong2(0ull, 0ull);
        for (ulonglong2& x : score) x = make_ulonglong2(0ull, 0ull);
    }
};

// A launch's tag is the number after the last launch's. One thread of every CTA takes it at its start; the last of them to have done so
// makes it the last one used, while the keys are under way: nothing is left for the end of the launch, for which the next one waits
// (the last CTA to leave counted itself out, stored and fenced: 2048 tokens, 2 heads 10.99 -> 10.21 us, 8192 15.4 -> 14.8, 4096 with 4 heads
// 13.1 -> 12.4). The last tag of all is the exception:
// at that launch's end words of old launches that were never written again are cleared (end_tags), before the tags start over at 1.
constexpr uint32_t kLastTag = 0xffffffffu;
__device__ __forceinline__ uint32_t take_tag(Exchange& x) {
    const uint32_t tag = ld_relaxed(&x.last_tag) + 1u;
    uint32_t old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(&x.started) : "memory");
    if (old + 1u == gridDim.x) {
        x.started = 0u;
        if (tag != kLastTag) x.last_tag = tag;
    }
    return tag;
}
// The tag as the CTA's other threads wait for it (bounded); 0: given up. It is mostly long there.
__device__ __forceinline__ uint32_t wait_tag(const volatile uint32_t* tag, volatile int* abort_flag) {
    uint32_t v;
    long long t0 = 0;
    for (uint32_t it = 1; (v = *tag) == 0u; ++it) {
        if (*abort_flag) return 0u;
        if ((it & 63u) == 0u) {
            if (t0 == 0) t0 = clock64();
            if (clock64() - t0 > kWaitLimitClocks) { *abort_flag = 1; return 0u; }
        }
    }
    return v;
}
__device__ __forceinline__ void end_tags(Exchange& x) {
    x.clear();
    x.last_tag = 0u;
}

}  // namespace chunkkv
