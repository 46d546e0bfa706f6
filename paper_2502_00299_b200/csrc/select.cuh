// Device-side bodies of the top-k chunk selection (ChunkKV Algorithm 3: "Top-K(chunk_scores, k)",
// the selection mask, "always keep most recent tokens", "nonzero(mask)"), shared by the
// stand-alone select kernel and the fused layer kernel. One CTA works on one KV head.
//
// Both bodies find the k-th largest of the order-preserving 32-bit keys exactly and then rank
// every chunk among the kept ones: rank = #above before it + min(#equal before it, ties to keep) -
// ties go to the lower chunk id. Token positions are written directly in ascending order: no
// mask, no sort.
//
// select_kept (keys in registers, or in shared memory where there are many a thread): an adaptive radix select
// (2048 equal sub-intervals of [min key, max key], repeated on the sub-interval that holds the k-th largest
// until few enough keys remain to rank directly).
//
// select_head_rows (keys nowhere or in a buffer of any kind; any number of kept chunks): 8 bits of the key at a time in
// short rolled loops. In the first
// pass every lane counts the four bins around the warp's first key in registers and the warp
// adds its totals once; any other bin, and every bin of the later passes, takes one
// shared-memory atomic per key.
//
// Keys in registers: a thread owns a run of consecutive ids. Otherwise each warp owns a contiguous block of chunk ids and walks
// it in rows of 32 consecutive ids, one per lane: accesses are coalesced and the order inside a row is the lane order; ranks
// come from warp ballots plus the warps' (#above, #equal) totals.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace chunkkv {

constexpr int kSelMaxWarps = 32;
constexpr int kSelCap = 8192;         // kept-chunk ids staged for coalesced index writes (16 bits each)
constexpr int kSelMaxChunks = 65535;  // most chunks of a head for which ids are staged

struct SelectSmem {
    alignas(16) unsigned short whist[kSelMaxWarps][256];
    alignas(16) unsigned short sel[kSelCap];
    int hist[256];
    unsigned long long warp_sums[kSelMaxWarps + 1];
    int warp_tot[kSelMaxWarps];
    uint32_t prefix;
    int need;
    int bin_count;
    int n_cand;
    int need_eq;
    int last_kept;
    alignas(16) int found[4];               // sub-interval of the k-th largest key, its rank in it, keys in it
    unsigned long long last;                // last candidate that is kept
};

__device__ __forceinline__ uint32_t select_order_key(float x) {
    const uint32_t b = __float_as_uint(x + 0.0f);          // -0 and +0 compare equal
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);     // larger float <=> larger key
}

// The one-CTA selection proper (select_regs, select_core; select_kept takes the one that fits): leaves the ids of the kept
// chunks in ascending order in sm.sel (kk = min(k, C) of them; kk <= kSelCap, C <= kSelMaxChunks) and sm.last_kept. All threads
// of the CTA must call this (it uses __syncthreads); blockDim.x must be a multiple of 32, at least 512 and at most 1024.
// sc2 != NULL: the head's scores are sc[ch] + sc2[ch] (a KV head scored as two heads of half the rows).
//
// The k-th largest key is found by an adaptive radix select: the keys of interest always lie in a
// known interval [base, base + span]; one round histograms them into 2048 equal sub-intervals,
// finds the sub-interval that holds the k-th largest and makes it the new interval. Chunk scores
// of one head sit in a narrow band of the float range, so the first round (over [min, max] of the
// keys) already leaves a handful of candidates; as soon as at most kSelCandCap keys remain they are
// ranked against each other directly. Ties and degenerate inputs (all keys equal) end with
// span = 0, i.e. a single key value. Exact for any input.
//
// What bounds it is a chain of latencies - seven or eight block-wide steps on a few thousand keys - and, inside the steps,
// the instructions that all warps issue. select_regs: a thread owns a run of KPT consecutive ids, so that a warp without
// ids leaves out the work on keys, loads are 8 or 16 bytes wide, and the order inside a warp is one prefix sum over its
// lanes. Candidates are ranked by (key, id) at once, so that ties need no counting of their own. select_core: registers with runs padded to four ids, or shared memory
// (warp v owns a block of consecutive ids and walks it in rows of 32, one id per lane, with ballots for the order); the ties are
// counted in a step more. In clocks, 576 threads, scores from the L2, a cold instruction cache, select_core -> select_regs: 204 keys
// 5.7k -> 4.0k, 816 5.5k -> 4.5k, 1636 6.0k -> 4.6k, 3274 6.6k -> 6.3k, 6550 15.0k -> 9.0k (runs padded to 16 ids were loaded one by
// one), 13104 20.2k (in shared memory) -> 14.8k. Then the last kept candidate was found first, so that one comparison a key and one
// prefix sum give the kept ids (two of each before), and four lanes rank a candidate: from the candidates' bin to the list 2.3k -> 1.8k
// clocks (204 and 819 keys); a layer of 2048 tokens, 2 heads 12.28 -> 11.84 us, of 8192 16.7 -> 16.3, of 32768 29.5 -> 29.2.
constexpr int kSelBins = 2048;
constexpr int kSelCandCap = 128;

// Scratch of a selection of k of C > k keys (every thread; before the barrier ahead of select_keys).
__device__ __forceinline__ void select_clear(SelectSmem& sm) {
    const int nt = blockDim.x, tid = threadIdx.x;
    if (tid == 0) { sm.last_kept = 0; sm.n_cand = 0; }
    for (int i = tid; i < kSelBins / 4; i += nt) reinterpret_cast<int4*>(&sm.whist[0][0])[i] = make_int4(0, 0, 0, 0);
    for (int i = tid; i < kSelCandCap; i += nt) reinterpret_cast<unsigned long long*>(&sm.sel[0])[i] = 0ull;
}
// k >= C or nothing to keep: no keys are needed. Every thread; true if that was it.
__device__ __forceinline__ bool select_all(int C, int k, SelectSmem& sm) {
    const int kk = min(k, C);
    if (k < C && kk > 0) return false;
    if (threadIdx.x == 0) sm.last_kept = kk > 0;
    for (int ch = threadIdx.x; ch < kk; ch += blockDim.x) sm.sel[ch] = static_cast<unsigned short>(ch);
    __syncthreads();
    return true;
}

// Keys in registers: thread t owns the ids [t KPT, (t + 1) KPT), C <= blockDim.x KPT; keys of ids past the last one are 0.
// Behind a barrier after select_clear and after every warp has left its smallest and largest key in sm.warp_sums.
template <int KPT>
__device__ __forceinline__ void select_keys(const uint32_t (&keys)[KPT], int C, int k, SelectSmem& sm) {
    constexpr unsigned kFull = 0xffffffffu;
    static_assert(KPT <= 32, "a run's flags fit a word");
    const int nt = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = nt >> 5;
    int* hist = reinterpret_cast<int*>(&sm.whist[0][0]);                            // kSelBins counters
    unsigned long long* cand = reinterpret_cast<unsigned long long*>(&sm.sel[0]);   // kSelCandCap keys with ids (sel is written later)
    const int id0 = tid * KPT, own = min(KPT, C - id0);      // this thread's ids; own <= 0: none
    const bool warp_on = warp * (32 * KPT) < C;              // this thread's warp has ids
    const unsigned long long mm = sm.warp_sums[lane < nwarps ? lane : 0];
    uint32_t base = __reduce_min_sync(kFull, static_cast<uint32_t>(mm));
    uint32_t span = __reduce_max_sync(kFull, static_cast<uint32_t>(mm >> 32)) - base;
    int need = k, n_bin = 0;        // the need-th largest of the n_bin keys in [base, base + span] is the k-th largest of all
    for (int round = 0;; ++round) {
        const int shift = max(0, 21 - __clz(span));          // (span >> shift) < kSelBins
        if (round > 0) {
            for (int i = tid; i < kSelBins / 4; i += nt) reinterpret_cast<int4*>(hist)[i] = make_int4(0, 0, 0, 0);
            __syncthreads();
        }
        if (warp_on) {
#pragma unroll
            for (int u = 0; u < KPT; ++u) {
                const uint32_t dlt = keys[u] - base;         // (a key below base wraps to more than span: base + span is a key's value)
                if (u < own && dlt <= span) atomicAdd(&hist[dlt >> shift], 1);
            }
        }
        __syncthreads();
        // thread t < 512 owns bins 2047 - 4t .. 2044 - 4t, so a prefix over threads counts from the top
        int cnt[4] = {0, 0, 0, 0}, sum = 0, inc = 0;
        if (tid < kSelBins / 4) {
            const int4 b4 = *reinterpret_cast<const int4*>(hist + kSelBins - 4 - 4 * tid);
            cnt[0] = b4.w; cnt[1] = b4.z; cnt[2] = b4.y; cnt[3] = b4.x;
            sum = (cnt[0] + cnt[1]) + (cnt[2] + cnt[3]);
            inc = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int n = __shfl_up_sync(kFull, inc, off);
                if (lane >= off) inc += n;
            }
            if (lane == 31) sm.warp_tot[warp] = inc;
        }
        __syncthreads();
        if (tid < kSelBins / 4) {
            inc += __reduce_add_sync(kFull, lane < warp ? sm.warp_tot[lane] : 0);
            if (inc - sum < need && need <= inc) {           // exactly one thread
                int ab = inc - sum, q = 0, cq = cnt[0];
#pragma unroll
                for (int t = 0; t < 3; ++t)                  // (unrolled: cnt stays in registers)
                    if (q == t && ab + cnt[t] < need) { ab += cnt[t]; q = t + 1; cq = cnt[t + 1]; }
                *reinterpret_cast<int4*>(&sm.found) = make_int4(kSelBins - 1 - 4 * tid - q, need - ab, cq, 0);
            }
        }
        __syncthreads();
        const int4 f = *reinterpret_cast<const int4*>(&sm.found);
        n_bin = f.z;
        need = f.y;
        const uint32_t sub = static_cast<uint32_t>(f.x) << shift;
        base += sub;
        span = min((1u << shift) - 1u, span - sub);
        if (n_bin <= kSelCandCap || span == 0u) break;
    }
    // The keys above the interval are kept, and `need` of those in it, the candidates. Few candidates: they are ranked against
    // each other by key and id, which gives the last one kept. Many equal ones: the first `need` of them in the order of ids.
    unsigned kept = 0;              // this thread's kept keys (bit u: id0 + u)
    int rank = 0;                   // kept keys before them
    if (n_bin <= kSelCandCap) {
        if (warp_on) {
            unsigned hits = 0;
#pragma unroll
            for (int u = 0; u < KPT; ++u) hits |= u < own && keys[u] - base <= span ? 1u << u : 0u;
            if (hits != 0) {                                     // (the order of the candidates does not matter)
                int at = atomicAdd(&sm.n_cand, __popc(hits));
#pragma unroll
                for (int u = 0; u < KPT; ++u)
                    if (hits >> u & 1u) cand[at++] = static_cast<unsigned long long>(keys[u]) << 32 | static_cast<uint32_t>(~(id0 + u));
            }
        }
        __syncthreads();
        if (warp * 8 < n_bin) {                                  // four lanes a candidate
            const int ci = tid >> 2;
            const unsigned long long v = ci < n_bin ? cand[ci] : 0ull;   // larger key first, then lower id: all different
            int gt = 0;
            const ulonglong2* c2 = reinterpret_cast<const ulonglong2*>(cand);
#pragma unroll 4
            for (int i = tid & 3; i < (n_bin + 1) / 2; i += 4) { const ulonglong2 x = c2[i]; gt += x.x > v; gt += x.y > v; }
            gt += __shfl_xor_sync(kFull, gt, 1);
            gt += __shfl_xor_sync(kFull, gt, 2);
            if ((tid & 3) == 0 && ci < n_bin && gt == need - 1) sm.last = v;
        }
        __syncthreads();
        if (warp_on) {
            const unsigned long long last = sm.last;
            const uint32_t last_key = static_cast<uint32_t>(last >> 32);
            const int last_id = static_cast<int>(~static_cast<uint32_t>(last));
#pragma unroll
            for (int u = 0; u < KPT; ++u)                        // (ids past the last one have key 0 and come behind every candidate)
                kept |= keys[u] > last_key || (keys[u] == last_key && id0 + u <= last_id) ? 1u << u : 0u;
            int total;
            if constexpr (KPT <= 4) {
                total = 0;
#pragma unroll
                for (int u = 0; u < KPT; ++u) {
                    const unsigned m = __ballot_sync(kFull, kept >> u & 1u);
                    rank += __popc(m & ((1u << lane) - 1u));
                    total += __popc(m);
                }
            } else {
                total = __popc(kept);
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int n = __shfl_up_sync(kFull, total, off);
                    if (lane >= off) total += n;
                }
                rank = total - __popc(kept);
            }
            if (lane == 31) sm.warp_tot[warp] = total;
        }
        __syncthreads();
        if (warp_on) rank += __reduce_add_sync(kFull, lane < warp ? sm.warp_tot[lane] : 0);
    } else {
        const uint32_t top = base + span;
        unsigned hits = 0;              // keys in the interval
        unsigned inc = 0, mine = 0;     // (#candidates << 16 | #above)
        if (warp_on) {
#pragma unroll
            for (int u = 0; u < KPT; ++u) {
                kept |= keys[u] > top ? 1u << u : 0u;
                hits |= u < own && keys[u] - base <= span ? 1u << u : 0u;
            }
            mine = __popc(kept) | __popc(hits) << 16;
            inc = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned n = __shfl_up_sync(kFull, inc, off);
                if (lane >= off) inc += n;
            }
            if (lane == 31) sm.warp_tot[warp] = static_cast<int>(inc);
        }
        __syncthreads();
        if (warp_on) {
            const unsigned ex = __reduce_add_sync(kFull, lane < warp ? static_cast<unsigned>(sm.warp_tot[lane]) : 0u) + inc - mine;
            const int eq_before = static_cast<int>(ex >> 16);
            rank = static_cast<int>(ex & 0xffffu) + min(eq_before, need);
            int room = max(0, need - eq_before);
#pragma unroll
            for (int u = 0; u < KPT; ++u)
                if (hits >> u & 1u) { kept |= room > 0 ? 1u << u : 0u; --room; }
        }
    }
    if (warp_on) {
#pragma unroll
        for (int u = 0; u < KPT; ++u)
            if (kept >> u & 1u) sm.sel[rank + __popc(kept & ((1u << u) - 1u))] = static_cast<unsigned short>(id0 + u);
        if (own > 0 && id0 + own == C && (kept >> (own - 1) & 1u)) sm.last_kept = 1;
    }
    __syncthreads();
}

// The same, keys from global memory.
template <int KPT>
__device__ __forceinline__ void select_regs(const float* sc, const float* sc2, int C, int k, SelectSmem& sm) {
    constexpr unsigned kFull = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (select_all(C, k, sm)) return;
    const int id0 = tid * KPT, own = min(KPT, C - id0);
    uint32_t keys[KPT];
    uint32_t lo = 0xffffffffu, hi = 0u;
    {
        float v[KPT];
        constexpr int W = KPT % 4 == 0 ? 4 : 2;              // floats a load
        auto load = [&](const float* p, float* o) {
            if constexpr (W == 4) {
                const float4 f = __ldcg(reinterpret_cast<const float4*>(p));
                o[0] = f.x; o[1] = f.y; o[2] = f.z; o[3] = f.w;
            } else {
                const float2 f = __ldcg(reinterpret_cast<const float2*>(p));
                o[0] = f.x; o[1] = f.y;
            }
        };
        const bool vec = ((reinterpret_cast<uintptr_t>(sc) | reinterpret_cast<uintptr_t>(sc2)) & (4u * W - 1u)) == 0;
        if (own == KPT && vec) {
#pragma unroll
            for (int u = 0; u < KPT; u += W) load(sc + id0 + u, &v[u]);
            if (sc2 != nullptr) {
                float v2[KPT];
#pragma unroll
                for (int u = 0; u < KPT; u += W) load(sc2 + id0 + u, &v2[u]);
#pragma unroll
                for (int u = 0; u < KPT; ++u) v[u] += v2[u];
            }
        } else if (own > 0) {
#pragma unroll
            for (int u = 0; u < KPT; ++u) v[u] = u < own ? __ldcg(sc + id0 + u) : 0.f;
            if (sc2 != nullptr) {
#pragma unroll
                for (int u = 0; u < KPT; ++u) v[u] += u < own ? __ldcg(sc2 + id0 + u) : 0.f;
            }
        }
        select_clear(sm);
        if (warp * (32 * KPT) < C) {
#pragma unroll
            for (int u = 0; u < KPT; ++u) {
                const bool in = u < own;
                keys[u] = in ? select_order_key(v[u]) : 0u;
                if (in) { lo = min(lo, keys[u]); hi = max(hi, keys[u]); }
            }
            lo = __reduce_min_sync(kFull, lo);
            hi = __reduce_max_sync(kFull, hi);
        }
    }
    if (lane == 0) sm.warp_sums[warp] = (static_cast<unsigned long long>(hi) << 32) | lo;
    __syncthreads();
    select_keys<KPT>(keys, C, k, sm);
}

// The same, keys in shared memory (16-byte aligned, room for a multiple of four behind the last one).
template <int KPT>
__device__ __forceinline__ void select_staged(const uint32_t* kbuf, int C, int k, SelectSmem& sm) {
    const int id0 = threadIdx.x * KPT;
    uint32_t keys[KPT];
    if (static_cast<int>(threadIdx.x >> 5) * (32 * KPT) < C) {
        constexpr int W = KPT % 4 == 0 ? 4 : 2;
#pragma unroll
        for (int u = 0; u < KPT; u += W) {
            if constexpr (W == 4) {
                const uint4 x = id0 + u < C ? *reinterpret_cast<const uint4*>(kbuf + id0 + u) : make_uint4(0u, 0u, 0u, 0u);
                keys[u] = x.x; keys[u + 1] = x.y; keys[u + 2] = x.z; keys[u + 3] = x.w;
            } else {
                const uint2 x = id0 + u < C ? *reinterpret_cast<const uint2*>(kbuf + id0 + u) : make_uint2(0u, 0u);
                keys[u] = x.x; keys[u + 1] = x.y;
            }
        }
#pragma unroll
        for (int u = 0; u < KPT; ++u)
            if (id0 + u >= C) keys[u] = 0u;
    }
    select_keys<KPT>(keys, C, k, sm);
}

// KPT > 0: up to KPT keys a thread in registers, in runs padded to four ids (C <= blockDim.x KPT; kbuf is not used). KPT = 0: the keys
// live in kbuf (shared memory, room for C).
template <int KPT>
__device__ __forceinline__ void select_core(const float* sc, const float* sc2, int C, int k, SelectSmem& sm, uint32_t* kbuf) {
    constexpr unsigned kFull = 0xffffffffu;
    constexpr bool REGS = KPT > 0;
    constexpr int UN = REGS ? KPT : 4;                       // unrolling of the loops over a warp's rows
    const int nt = blockDim.x, nwarps = nt >> 5;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool keep_all = (k >= C);
    const int kk = min(k, C);
    // registers: thread t owns the ids [t per, (t + 1) per); shared memory: lane l of warp v the ids id0 + 32 u, u < per
    const int per = REGS ? 4 * ((C + 4 * nt - 1) / (4 * nt)) : (C + nt - 1) / nt;
    const int rows = REGS ? KPT : per;
    const int id0 = REGS ? tid * per : warp * per * 32 + lane;
    const int own = REGS ? max(0, min(per, C - id0)) : 0;    // ids of this thread
    uint32_t keys[REGS ? KPT : 1];
    auto have = [&](int u) { return REGS ? u < own : (u < per && id0 + 32 * u < C); };
    auto key_at = [&](int u) -> uint32_t { return REGS ? keys[REGS ? u : 0] : kbuf[id0 + 32 * u]; };

    if (tid == 0) { sm.last_kept = 0; sm.n_cand = 0; }
    uint32_t thresh = 0;   // key of the k-th largest score
    int need_eq = 0;       // how many chunks equal to the threshold are kept
    if (!keep_all && kk > 0) {
        int* hist = reinterpret_cast<int*>(&sm.whist[0][0]);            // kSelBins counters
        uint32_t* cand = reinterpret_cast<uint32_t*>(&sm.sel[0]);       // kSelCandCap keys (sel is written later)
        uint32_t lo = 0xffffffffu, hi = 0u;
        if constexpr (REGS) {
            float v[KPT];                                    // (all loads before the first use)
            const bool vec = ((reinterpret_cast<uintptr_t>(sc) | reinterpret_cast<uintptr_t>(sc2)) & 15u) == 0 && own == KPT;
            if (vec) {
#pragma unroll
                for (int u = 0; u < KPT; u += 4) {
                    const float4 f = __ldcg(reinterpret_cast<const float4*>(sc + id0 + u));
                    v[u] = f.x; v[u + 1] = f.y; v[u + 2] = f.z; v[u + 3] = f.w;
                }
                if (sc2 != nullptr) {
#pragma unroll
                    for (int u = 0; u < KPT; u += 4) {
                        const float4 f = __ldcg(reinterpret_cast<const float4*>(sc2 + id0 + u));
                        v[u] += f.x; v[u + 1] += f.y; v[u + 2] += f.z; v[u + 3] += f.w;
                    }
                }
            } else {
#pragma unroll
                for (int u = 0; u < KPT; ++u) v[u] = have(u) ? __ldcg(sc + id0 + u) : 0.f;
                if (sc2 != nullptr) {
#pragma unroll
                    for (int u = 0; u < KPT; ++u) v[u] += have(u) ? __ldcg(sc2 + id0 + u) : 0.f;
                }
            }
            for (int i = tid; i < kSelBins; i += nt) hist[i] = 0;
#pragma unroll
            for (int u = 0; u < KPT; ++u) {
                keys[u] = select_order_key(v[u]);
                if (have(u)) { lo = min(lo, keys[u]); hi = max(hi, keys[u]); }
            }
        } else {
            for (int i = tid; i < kSelBins; i += nt) hist[i] = 0;
            constexpr int kB = 16;                           // loads in flight per thread
#pragma unroll 1
            for (int u0 = 0; u0 < rows; u0 += kB) {
                float v[kB];
#pragma unroll
                for (int q = 0; q < kB; ++q) v[q] = __ldcg(sc + min(id0 + 32 * min(u0 + q, rows - 1), C - 1));
                if (sc2 != nullptr) {
#pragma unroll
                    for (int q = 0; q < kB; ++q) v[q] += __ldcg(sc2 + min(id0 + 32 * min(u0 + q, rows - 1), C - 1));
                }
#pragma unroll
                for (int q = 0; q < kB; ++q)
                    if (have(u0 + q)) {
                        const uint32_t key = select_order_key(v[q]);
                        kbuf[id0 + 32 * (u0 + q)] = key;     // (read back by this thread only)
                        lo = min(lo, key);
                        hi = max(hi, key);
                    }
            }
        }
        lo = __reduce_min_sync(kFull, lo);
        hi = __reduce_max_sync(kFull, hi);
        if (lane == 0) sm.warp_sums[warp] = (static_cast<unsigned long long>(hi) << 32) | lo;
        __syncthreads();
        // smallest and largest key of the head
        const unsigned long long mm = sm.warp_sums[lane < nwarps ? lane : 0];
        uint32_t base = __reduce_min_sync(kFull, static_cast<uint32_t>(mm));
        uint32_t span = __reduce_max_sync(kFull, static_cast<uint32_t>(mm >> 32)) - base;   // the keys of interest lie in [base, base + span]
        int need = k;                        // the need-th largest of them is the threshold
        for (int round = 0;; ++round) {
            if (span == 0u) { thresh = base; need_eq = need; break; }
            const int shift = max(0, 21 - __clz(span));      // (span >> shift) < kSelBins
            if (round > 0) {
                for (int i = tid; i < kSelBins; i += nt) hist[i] = 0;
                __syncthreads();
            }
#pragma unroll UN
            for (int u = 0; u < rows; ++u)
                if (have(u)) {
                    const uint32_t dlt = key_at(u) - base;   // (a key below base wraps to more than span: base + span is a key's value)
                    if (dlt <= span) atomicAdd(&hist[dlt >> shift], 1);
                }
            __syncthreads();
            // thread t < 512 owns bins 2047 - 4t .. 2044 - 4t, so a prefix over threads counts from the top
            int cnt[4] = {0, 0, 0, 0};
            if (tid < kSelBins / 4) {
                const int4 b4 = *reinterpret_cast<const int4*>(hist + kSelBins - 4 - 4 * tid);
                cnt[0] = b4.w; cnt[1] = b4.z; cnt[2] = b4.y; cnt[3] = b4.x;
            }
            const int sum = (cnt[0] + cnt[1]) + (cnt[2] + cnt[3]);
            int inc = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int n = __shfl_up_sync(kFull, inc, off);
                if (lane >= off) inc += n;
            }
            if (lane == 31) sm.warp_tot[warp] = inc;
            __syncthreads();
            inc += __reduce_add_sync(kFull, lane < warp ? sm.warp_tot[lane] : 0);
            if (tid < kSelBins / 4 && inc - sum < need && need <= inc) {     // exactly one thread
                int above = inc - sum, q = 0, cq = cnt[0];
#pragma unroll
                for (int t = 0; t < 3; ++t)          // (unrolled: cnt stays in registers)
                    if (q == t && above + cnt[t] < need) { above += cnt[t]; q = t + 1; cq = cnt[t + 1]; }
                sm.prefix = static_cast<uint32_t>(kSelBins - 1 - 4 * tid - q);
                sm.need = need - above;
                sm.bin_count = cq;
            }
            __syncthreads();
            const uint32_t bin = sm.prefix;
            const int n_bin = sm.bin_count;
            need = sm.need;
            const uint32_t sub = bin << shift;
            base += sub;
            span = min((1u << shift) - 1u, span - sub);
            if (n_bin <= kSelCandCap) {
                // few keys left: rank them against each other
                if constexpr (REGS) {
                    unsigned hits = 0;
#pragma unroll
                    for (int u = 0; u < KPT; ++u) hits |= (have(u) && keys[u] - base <= span) ? 1u << u : 0u;
                    if (hits != 0) {
                        int at = atomicAdd(&sm.n_cand, __popc(hits));
#pragma unroll
                        for (int u = 0; u < KPT; ++u)
                            if (hits >> u & 1u) cand[at++] = keys[u];
                    }
                } else {
#pragma unroll 4
                    for (int u = 0; u < rows; ++u)
                        if (have(u) && key_at(u) - base <= span) cand[atomicAdd(&sm.n_cand, 1)] = key_at(u);
                }
                __syncthreads();
                if (tid < n_bin) {
                    const uint32_t v = cand[tid];
                    int gt = 0, ge = 0;
#pragma unroll 8
                    for (int i = 0; i < n_bin; ++i) { const uint32_t x = cand[i]; gt += x > v; ge += x >= v; }
                    if (gt < need && need <= ge) { sm.prefix = v; sm.need_eq = need - gt; }   // same values from every writer
                }
                __syncthreads();
                thresh = sm.prefix;
                need_eq = sm.need_eq;
                break;
            }
        }
    }

    // Ordered sweep over the chunk ids: a kept chunk's rank is the number of kept ones before it, (#above) + min(#equal,
    // ties to keep). (#equal << 16 | #above) of a thread or warp fits 32 bits, and so do the totals: fewer than k keys lie
    // above the threshold, C <= kSelMaxChunks.
    if (kk > 0 && keep_all) {
        for (int ch = tid; ch < C; ch += nt) sm.sel[ch] = static_cast<unsigned short>(ch);
        if (tid == 0) sm.last_kept = 1;
    } else if (kk > 0 && REGS) {
        unsigned mine = 0;
#pragma unroll
        for (int u = 0; u < KPT; ++u) mine += have(u) ? (keys[u] > thresh ? 1u : (keys[u] == thresh ? 0x10000u : 0u)) : 0u;
        unsigned inc = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned n = __shfl_up_sync(kFull, inc, off);
            if (lane >= off) inc += n;
        }
        if (lane == 31) sm.warp_tot[warp] = static_cast<int>(inc);
        __syncthreads();                 // (also: cand, which shares its words with sel, is no longer read)
        inc += __reduce_add_sync(kFull, lane < warp ? static_cast<unsigned>(sm.warp_tot[lane]) : 0u) - mine;
        int eq_before = static_cast<int>(inc >> 16);
        int rank = static_cast<int>(inc & 0xffffu) + min(eq_before, need_eq);
#pragma unroll
        for (int u = 0; u < KPT; ++u) {
            const bool eq = have(u) && keys[u] == thresh;
            const bool kept = have(u) && (keys[u] > thresh || (eq && eq_before < need_eq));
            if (kept) sm.sel[rank] = static_cast<unsigned short>(id0 + u);
            if (kept && id0 + u == C - 1) sm.last_kept = 1;
            rank += kept;
            eq_before += eq;
        }
    } else if (kk > 0) {
        const unsigned lt_mask = (1u << lane) - 1u;
        unsigned gt_n = 0, eq_n = 0;
#pragma unroll 4
        for (int u = 0; u < rows; ++u) {
            const uint32_t key = have(u) ? key_at(u) : 0u;
            gt_n += __popc(__ballot_sync(kFull, have(u) && key > thresh));
            eq_n += __popc(__ballot_sync(kFull, have(u) && key == thresh));
        }
        if (lane == 0) sm.warp_tot[warp] = static_cast<int>(eq_n << 16 | gt_n);
        __syncthreads();                 // (also: cand, which shares its words with sel, is no longer read)
        const unsigned tot = __reduce_add_sync(kFull, lane < warp ? static_cast<unsigned>(sm.warp_tot[lane]) : 0u);
        unsigned gt_run = tot & 0xffffu, eq_run = tot >> 16;
#pragma unroll 4
        for (int u = 0; u < rows; ++u) {
            const uint32_t key = have(u) ? key_at(u) : 0u;
            const bool gt = have(u) && key > thresh, eq = have(u) && key == thresh;
            const unsigned gtm = __ballot_sync(kFull, gt), eqm = __ballot_sync(kFull, eq);
            const int gt_before = gt_run + __popc(gtm & lt_mask);
            const int eq_before = eq_run + (eqm ? __popc(eqm & lt_mask) : 0);
            if (gt || (eq && eq_before < need_eq)) {
                sm.sel[gt_before + min(eq_before, need_eq)] = static_cast<unsigned short>(id0 + 32 * u);
                if (id0 + 32 * u == C - 1) sm.last_kept = 1;
            }
            gt_run += __popc(gtm);
            eq_run += eqm ? __popc(eqm) : 0;
        }
    }
    __syncthreads();
}

// The selection, by the number of keys a thread has to take; kbuf: room for C keys in shared memory, used beyond
// select_reg_keys() keys a thread. select.cu and the layer kernel's wide variant take select_regs up to there (the layer kernel takes its keys from
// shared memory otherwise: select_staged). The other kernels have no registers
// to spare beside their own: with select_regs for 6 keys or more the model kernel spills and a call with 5994 chunks is 8 %
// slower, so it takes that form up to 4 keys a thread (32 layers of 4096 tokens 348 -> 311 us, 16 layers of 20000 tokens in chunks
// of 16 228 -> 206); the kernels of score.cu spill with any of it, and so does the model kernel's big variant for chunks of 8 (30 bytes
// a thread instead of 28; 12000 tokens, 224 rows 303 -> 308 us, 24000 tokens, 256 rows 270 -> 279; the big variants of the other sizes are 0.5 to
// 2 % faster with it).
// What else is compiled into a kernel changes how its scoring loops are scheduled, without a spill: the layer kernel with the bodies for more
// than 16 keys a thread beside the others is slower at 80000 tokens (28 query heads, 112 rows, chunks of 32 35.7 -> 36.6 us), so those are a variant of
// it.
// (All inlined: as a function its register convention made the kernels' scoring loops spill, 2 to 10 % of a model call; the layer
// kernel does not spill with it, but is 1 to 2 % slower.)
enum SelectIn {
    kSelScratch,        // the kernels of score.cu
    kSelModel,          // the model kernel
    kSelModelCore,      // the same without select_regs
    kSelLayer,          // the layer kernel, at most 16 keys a thread (select_staged, not select_kept)
    kSelLayerWide,      // the layer kernel, more
    kSelAlone           // select.cu
};
__host__ __device__ constexpr int select_reg_keys(SelectIn where) {
    return where == kSelLayerWide || where == kSelAlone ? 24 : (where == kSelScratch ? 8 : 16);
}

template <SelectIn WHERE>
__device__ __forceinline__ void select_kept(const float* sc, const float* sc2, int C, int k, SelectSmem& sm, uint32_t* kbuf) {
    static_assert(WHERE != kSelLayer, "takes its keys from shared memory");
    const int per = (C + static_cast<int>(blockDim.x) - 1) / static_cast<int>(blockDim.x);
    if (per > select_reg_keys(WHERE)) return select_core<0>(sc, sc2, C, k, sm, kbuf);
    if constexpr (WHERE == kSelModel || WHERE == kSelAlone) {
        // the shortest run that covers the ids: the longer ones leave more warps without any, and a step's time goes with the
        // keys of the busiest scheduler (816 keys: runs of 2 4.5k clocks, of 4 5.2k; 1636 keys: of 4 4.6k, of 8 5.7k)
        if (per <= 2) return select_regs<2>(sc, sc2, C, k, sm);
        if (per <= 4) return select_regs<4>(sc, sc2, C, k, sm);
    }
    if constexpr (WHERE == kSelAlone) {
        if (per <= 8) return select_regs<8>(sc, sc2, C, k, sm);
        if (per <= 16) return select_regs<16>(sc, sc2, C, k, sm);
    }
    if constexpr (WHERE == kSelLayerWide || WHERE == kSelAlone) {
        select_regs<24>(sc, sc2, C, k, sm);
    } else {
        if (WHERE == kSelScratch || per <= 8) return select_core<8>(sc, sc2, C, k, sm, nullptr);
        if constexpr (WHERE != kSelScratch) select_core<16>(sc, sc2, C, k, sm, nullptr);
    }
}

// Tokens of the kept chunks that are emitted: every kept chunk is full except possibly chunk C - 1, which can only be
// the last kept one. tok_cap: at most this many, lowest positions first (Algorithm 1 keeps the first L_max - w
// selected tokens); no cap by default.
__device__ __forceinline__ int select_tokens(int P, int c, int C, int k, const SelectSmem& sm, int tok_cap = 0x7fffffff) {
    const int kk = min(k, C);
    const int tail = (C > 0) ? (P - (C - 1) * c) : 0;
    return min(kk * c - ((sm.last_kept && kk > 0) ? (c - tail) : 0), tok_cap);
}

// Kept position n of [0, n_max): tokens of the kept chunks ascending, then the window, then -1.
__device__ __forceinline__ int select_position(const SelectSmem& sm, int n, int n_tok, int c, int P, int w) {
    if (n < n_tok) { const int r = n / c; return sm.sel[r] * c + (n - r * c); }
    return n < n_tok + w ? P + (n - n_tok) : -1;
}

// The whole selection of a head into out[n_max]; conditions as select_kept.
template <SelectIn WHERE>
__device__ __forceinline__ void select_head(const float* sc, const float* sc2, int L, int w, int c, int C, int k, int n_max,
                                            int32_t* out, SelectSmem& sm, uint32_t* kbuf, int tok_cap = 0x7fffffff) {
    select_kept<WHERE>(sc, sc2, C, k, sm, kbuf);
    const int P = L - w, n_tok = select_tokens(P, c, C, k, sm, tok_cap);
    for (int n = threadIdx.x; n < n_max; n += blockDim.x) out[n] = select_position(sm, n, n_tok, c, P, w);
    __syncthreads();     // shared state may be reused by the caller
}

// Selection for many chunks per thread. All threads of the CTA must call this (it uses
// __syncthreads); blockDim.x must be a multiple of 32 and at most 1024. kbuf: room for C keys
// (shared or global memory; it may be the score array itself, which is then overwritten), or
// NULL: keys are then recomputed from the scores on every use. sc2 != NULL: the head's scores are sc[ch] + sc2[ch] (a KV head scored as two
// heads of half the rows).
__device__ __forceinline__ void select_head_rows(const float* sc, const float* sc2, int L, int w, int c, int C, int k,
                                            int n_max, int32_t* __restrict__ out, SelectSmem& sm, uint32_t* kbuf,
                                            int tok_cap = 0x7fffffff) {
    auto score_at = [&](int ch) { return sc2 != nullptr ? __ldcg(sc + ch) + __ldcg(sc2 + ch) : __ldcg(sc + ch); };
    constexpr unsigned kFull = 0xffffffffu;
    const int P = L - w;
    const int nt = blockDim.x, nwarps = nt >> 5;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    const bool keep_all = (k >= C);
    const int kk = min(k, C);

    // warp v owns chunk ids [v * rows * 32, (v + 1) * rows * 32); row u of it holds base + 32 u (+ lane)
    const int rows = (C + nt - 1) / nt;
    const int base = warp * rows * 32 + lane;
    const bool need_keys = kk > 0 && !keep_all;
    if (need_keys && kbuf != nullptr) {
        // kB loads in flight per thread, no control flow between them (ids past the end are clamped)
        constexpr int kB = 16;
#pragma unroll 1
        for (int ch0 = tid; ch0 < C; ch0 += kB * nt) {
            float v[kB];
#pragma unroll
            for (int q = 0; q < kB; ++q) v[q] = __ldcg(sc + min(ch0 + q * nt, C - 1));
            if (sc2 != nullptr) {
#pragma unroll
                for (int q = 0; q < kB; ++q) v[q] += __ldcg(sc2 + min(ch0 + q * nt, C - 1));
            }
#pragma unroll
            for (int q = 0; q < kB; ++q)
                if (ch0 + q * nt < C) kbuf[ch0 + q * nt] = select_order_key(v[q]);
        }
    }
    if (tid == 0) sm.last_kept = 0;
    __syncthreads();                                         // kbuf complete
    auto key_at = [&](int ch) -> uint32_t { return kbuf != nullptr ? kbuf[ch] : select_order_key(score_at(ch)); };

    uint32_t thresh = 0;   // key of the k-th largest score
    int need_eq = 0;       // how many chunks equal to the threshold are kept
    if (need_keys) {
        uint32_t prefix = 0;
        int need = k;
#pragma unroll 1
        for (int pass = 0; pass < 4; ++pass) {
            const int shift = 24 - 8 * pass;
            if (tid < 256) sm.hist[tid] = 0;
            __syncthreads();
            if (pass == 0) {
                // bins b0 - 1 .. b0 + 2 around the bin of the warp's first key are counted in
                // registers (two 16-bit counters per register; a lane sees at most `rows` keys)
                const int ch_first = warp * rows * 32;
                const int b0 = (ch_first < C) ? static_cast<int>(key_at(ch_first) >> 24) : 0;
                const bool packed = rows < 65536;
                uint32_t lo = 0u, hi = 0u;
#pragma unroll 4
                for (int u = 0; u < rows; ++u) {
                    const int ch = base + 32 * u;
                    if (ch < C) {
                        const int bin = static_cast<int>(key_at(ch) >> 24);
                        const unsigned d = static_cast<unsigned>(bin - b0 + 1);
                        if (packed && d < 4u) {
                            const uint32_t inc = 1u << ((d & 1u) * 16u);
                            lo += (d < 2u) ? inc : 0u;
                            hi += (d < 2u) ? 0u : inc;
                        } else {
                            atomicAdd(&sm.hist[bin], 1);
                        }
                    }
                }
                const unsigned c0 = __reduce_add_sync(kFull, lo & 0xffffu), c1 = __reduce_add_sync(kFull, lo >> 16);
                const unsigned c2 = __reduce_add_sync(kFull, hi & 0xffffu), c3 = __reduce_add_sync(kFull, hi >> 16);
                if (lane == 0) {   // a non-zero count belongs to a bin some key fell into: 0 <= bin <= 255
                    if (c0) atomicAdd(&sm.hist[b0 - 1], static_cast<int>(c0));
                    if (c1) atomicAdd(&sm.hist[b0], static_cast<int>(c1));
                    if (c2) atomicAdd(&sm.hist[b0 + 1], static_cast<int>(c2));
                    if (c3) atomicAdd(&sm.hist[b0 + 2], static_cast<int>(c3));
                }
            } else {
                const uint32_t himask = 0xFFFFFFFFu << (shift + 8);
#pragma unroll 4
                for (int u = 0; u < rows; ++u) {
                    const int ch = base + 32 * u;
                    if (ch < C) {
                        const uint32_t key = key_at(ch);
                        if ((key & himask) == prefix) atomicAdd(&sm.hist[(key >> shift) & 0xFFu], 1);
                    }
                }
            }
            __syncthreads();
            if (warp == 0) {
                // lane t owns bins 255-8t .. 248-8t (descending), so a prefix over lanes counts from the top
                int cnt[8], sum = 0;
#pragma unroll
                for (int q = 0; q < 8; ++q) { cnt[q] = sm.hist[255 - 8 * lane - q]; sum += cnt[q]; }
                int inc = sum;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int n = __shfl_up_sync(kFull, inc, off);
                    if (lane >= off) inc += n;
                }
                const unsigned reach = __ballot_sync(kFull, inc >= need);
                const int owner = reach ? (__ffs(reach) - 1) : 31;
                if (lane == owner) {
                    int above = inc - sum, q = 0;
                    while (q < 7 && above + cnt[q] < need) { above += cnt[q]; ++q; }
                    sm.prefix = prefix | (static_cast<uint32_t>(255 - 8 * lane - q) << shift);
                    sm.need = need - above;
                }
            }
            __syncthreads();
            prefix = sm.prefix;
            need = sm.need;
        }
        thresh = prefix;
        need_eq = need;
    }

    // Ordered sweep over the chunk ids: ballots give a row's (#above, #equal) in lane order.
    const bool stage_sel = kk <= kSelCap && C <= kSelMaxChunks;
    if (kk > 0) {
        auto row_flags = [&](int ch, unsigned& gtm, unsigned& eqm, bool& gt, bool& eq) {
            const bool valid = ch < C;
            uint32_t key = 0u;
            if (!keep_all && valid) key = key_at(ch);
            gt = valid && (keep_all || key > thresh);
            eq = valid && !keep_all && key == thresh;
            gtm = __ballot_sync(kFull, gt);
            eqm = __ballot_sync(kFull, eq);
        };
        unsigned gt_n = 0, eq_n = 0;                         // the warp's totals (same in every lane)
#pragma unroll 4
        for (int u = 0; u < rows; ++u) {
            unsigned gtm, eqm;
            bool gt, eq;
            row_flags(base + 32 * u, gtm, eqm, gt, eq);
            gt_n += __popc(gtm);
            eq_n += __popc(eqm);
        }
        // block-wide exclusive prefix of the packed pair (eq in the high half, gt in the low half)
        if (lane == 0) sm.warp_sums[warp] = (static_cast<unsigned long long>(eq_n) << 32) | gt_n;
        __syncthreads();
        if (warp == 0) {
            const unsigned long long s = (lane < nwarps) ? sm.warp_sums[lane] : 0ull;
            unsigned long long sinc = s;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned long long n = __shfl_up_sync(kFull, sinc, off);
                if (lane >= off) sinc += n;
            }
            sm.warp_sums[lane] = sinc - s;
        }
        __syncthreads();
        const unsigned long long excl = sm.warp_sums[warp];
        int gt_run = static_cast<int>(excl & 0xffffffffu), eq_run = static_cast<int>(excl >> 32);
#pragma unroll 2
        for (int u = 0; u < rows; ++u) {
            const int ch = base + 32 * u;
            unsigned gtm, eqm;
            bool gt, eq;
            row_flags(ch, gtm, eqm, gt, eq);
            const int gt_before = gt_run + __popc(gtm & lt_mask);
            const int eq_before = eq_run + __popc(eqm & lt_mask);
            if (gt || (eq && eq_before < need_eq)) {
                const int rank = gt_before + min(eq_before, need_eq);
                if (stage_sel) sm.sel[rank] = static_cast<unsigned short>(ch);
                else {
                    const int j0 = ch * c, len = min(c, P - j0);
                    int32_t* dst = out + static_cast<size_t>(rank) * c;
                    for (int t = 0; t < len; ++t)
                        if (rank * c + t < tok_cap) dst[t] = j0 + t;
                }
                if (ch == C - 1) sm.last_kept = 1;
            }
            gt_run += __popc(gtm);
            eq_run += __popc(eqm);
        }
    }
    __syncthreads();
    // Every kept chunk is full except possibly chunk C-1, which can only be the last kept one.
    const int tail = (C > 0) ? (P - (C - 1) * c) : 0;
    // tok_cap: at most this many tokens of the kept chunks are emitted, lowest positions first
    // (Algorithm 1 keeps the first L_max - w selected tokens); no cap by default
    const int n_tok = min(kk * c - ((sm.last_kept && kk > 0) ? (c - tail) : 0), tok_cap);
    if (stage_sel)
        for (int n = tid; n < n_tok; n += nt) {
            const int rank = n / c;
            out[n] = sm.sel[rank] * c + (n - rank * c);
        }
    for (int i = tid; i < w; i += nt) out[n_tok + i] = P + i;
    for (int i = n_tok + w + tid; i < n_max; i += nt) out[i] = -1;
    __syncthreads();     // shared state may be reused by the caller
}

}  // namespace chunkkv
