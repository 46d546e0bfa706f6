// The whole layer in one launch with the chunk partial sums kept on chip
// (ChunkKV Algorithm 3: observe-window scores, chunk scores, top-k, index_select on K and V).
//
// Every CTA belongs to one scoring head and owns a contiguous range of its keys. While it streams its
// keys through the tensor cores it keeps, per query row and chunk, the sum of exp2(s - m_panel) in
// TENSOR MEMORY (lane = query row, column = chunk of the CTA's range, 256 columns beside the two
// accumulator buffers) and the panel maxima in shared memory, so for most shapes nothing but a
// (max, sum) pair per row and CTA goes to global memory before the chunk scores themselves. A key
// range with more panels than those 256 columns hold (long contexts, small chunks) keeps the rest
// in scratch (L2): written and read back by the same thread, 16 bytes at a time.
//
// A KV head is one scoring head where it has at most 128 query rows. With more, one of two forms:
//   - two scoring heads of half the rows each, with half the CTAs each, where all their panels stay on chip; the two
//     vectors of chunk scores are added in the selection;
//   - two query tiles, scored by the same CTAs: each key tile is loaded once and multiplied with both, and the two pairs
//     of epilogue groups take one query tile each; with one query tile the pairs take alternate key tiles. In both cases
//     the CTA's products are numbered in issue order ("virtual tiles"), accumulator and pair = number modulo 2, so one set
//     of loops serves both.
// Two heads are the faster form wherever their panels stay on chip (device times, two tiles -> two heads; 64 heads over 8,
// c = 10: 1024 tokens 15.8 -> 13.9 us, 4096 18.3 -> 16.5, 10248 22.7 -> 20.8, 20480 31.0 -> 29.2; c = 20, 45000 tokens 50.5 -> 48.9;
// 16 over 2, 8192 tokens 18.2 -> 15.6): a CTA has half the exponentials to do between the latencies of its chain, twice as
// many CTAs gather, and K's second reading is an L2 hit. Past that the partial sums in scratch would double as well.
//
// What bounds it (8 KV heads, d 128, B200): up to 128 rows the DRAM stream of K while scoring (12 of
// 28.6 us on the device at 32K tokens, c = 10) and then a chain of latencies (two hand-overs, selection, gather);
// beyond 128 rows the special-function unit (one exponential per score element, 16 per clock and
// SM: 80 % of that rate while scoring; 86 % is what this pipeline reaches with nothing else to do). Against the kernel of score.cu, which keeps every partial sum
// in scratch, loads K once per query tile and takes run-time chunk sizes: c = 16, 32768 tokens, 256 rows
// 121 -> 41 us; c = 20, 131072 tokens, 256 rows 161 -> 139 us; chunk scores alone (c = 10, 32768
// tokens, 128 rows, four launches) 32 -> 20 us.
//
//   1. score      TMA -> tcgen05.mma (128 rows x 120 or 128 keys per accumulator tile) -> epilogue
//                 warps: one exponential per score element, chunk sums to tensor memory
//   2. hand-over  the CTAs of a scoring head publish their per-row (max, sum) and take one another's: words that carry
//                 the launch's tag beside the value, or (lanes) a per-head counter (bounded waits)
//   3. contract   every CTA merges the head's records into m_i and 1 / l_i and contracts its own
//                 partial sums over the rows: chunk scores of its key range -> global memory
//   4. hand-over  per KV head, until all of its chunk scores are there (tagged words or a counter, bounded wait)
//   5. select     every CTA of the KV head runs the same exact top-k over the head's chunk scores
//                 and so holds the kept chunks in shared memory without a third wait
//   6. gather     the head's output positions are split evenly over its CTAs: each expands its
//                 share to token positions, writes them to out_idx and moves their rows
//
// Without out_idx the kernel ends after step 3 (chunk scores are the result).
//
// Heads never wait for each other. All CTAs of a launch are resident while they wait for their head's other CTAs: at
// most one per SM, and a cooperative launch where several launches share the GPU (lanes); every wait gives up after a
// clock limit, raises the device status word and lets the CTA leave.
#include "gather.cuh"
#include "internal.h"
#include "panels.cuh"
#include "ptx.cuh"
#include "resident.cuh"
#include "select.cuh"

#include <math_constants.h>

namespace chunkkv {

namespace {

constexpr int kRThreads = 576;               // warp 0: TMA, warp 1: UMMA issue, warps 2..17: epilogue
constexpr int kRMiscBytes = 10240;           // records of the four epilogue groups, slices, m_i, 1 / l_i

struct ResCtl {
    unsigned long long full[kRMaxStages];
    unsigned long long empty[kRMaxStages];
    unsigned long long tfull[2];
    unsigned long long tempty[2];
    unsigned long long qfull;
    int rec_count[2][4];               // epilogue warps that have left their part of the CTA's record: [query tile][32 rows]
    uint32_t tmem_base;
    uint32_t tag;                      // this launch's tag (0: not known yet)
    int abort_flag;
    int wait_ok;
};

__device__ Exchange g_exchange[kExchangeSlots];
enum { kDirectRecords = 1, kDirectScores = 2 };

// After scoring the ring holds the selection's scratch, then the head's keys if they fit. A CTA lists the head's kept chunks where the
// list has room for them and, but for the wide variant, a thread takes all of its keys at once; else it works on the scores in global
// memory. Chunk scores go through the exchange only where every CTA lists, so the host asks the same function as the kernel.
constexpr size_t kRSelBytes = (sizeof(SelectSmem) + 127) & ~size_t(127);
__host__ __device__ constexpr bool keys_fit(int C, int ring_bytes) {
    return kRSelBytes + (static_cast<size_t>(C) + 4) * 4 <= static_cast<size_t>(ring_bytes);
}
__host__ __device__ constexpr bool lists_kept(bool wide, int C, int k, int ring_bytes) {
    return (k < C ? k : C) <= kSelCap && C <= kSelMaxChunks && keys_fit(C, ring_bytes) && (wide || C <= kRThreads * select_reg_keys(kSelLayer));
}

struct ResArgs {
    int L, P, w, R, d;                 // R rows per KV head
    short n_mt;                        // 128-row query tiles per KV head (1 or 2)
    short shift;                       // 1: the rows of a KV head are scored as two heads of q_rows and the rest
    int direct;                        // hand-overs that go through the exchange
    int q_rows;                        // rows of a box of the query tensor map: 128, fewer, or the half's
    float sl2;                         // log2(e) / sqrt(d)
    int cph;                           // CTAs per scoring head (a KV head, or one of its halves)
    int n_stages;
    int k, n_max, Hkv;
    int off_ring, ring_bytes, off_pmax, off_misc;   // dynamic shared memory layout (bytes from the aligned base)
    int n_on, n_off;                   // panels of a CTA kept on chip; room for panels in scratch
    int spill_rows;                    // rows of a panel's record in scratch
    const uint4* K;
    const uint4* V;
    long long k_row, k_head, v_row, v_head;   // 16-byte vectors between rows of a head / between heads
    const int32_t* block_table;              // non-null: out_K / out_V are paged caches
    int page_size, num_pages;
    int tok_cap;                             // Algorithm 1: tokens of the kept chunks that are emitted
    uint4* out_K;
    uint4* out_V;
    int32_t* out_idx;
    union {
        float* cta_stat;               // [grid, n_mt, {max, sum}, 128] (hand-over by counters)
        Exchange* x;                   // (direct != 0)
    };
    float* scores;                     // [Hkv, score_row]
    int score_row;                     // C, or C rounded up to a multiple of 4 in scratch (16-byte aligned rows)
    float* spill;                      // [grid, n_off, (chunk slots per panel + 1) * spill_rows]: chunk sums, panel maximum
    unsigned* counters;                // header + kResidentCountersOffset, zero between launches

    __device__ unsigned* exits() const { return counters; }              // CTAs that left; the last one clears the counters
    __device__ unsigned* cnt_a(int h) const { return counters + 16 + h; }                          // hand-over 2 of a scoring head
    __device__ unsigned* cnt_b(int h) const { return counters + 16 + kResidentMaxHeads + h; }      // hand-over 4 of a KV head
    __device__ int* status() const { return reinterpret_cast<int*>(counters) - kResidentCountersOffset / sizeof(int); }
};
// A launch that comes between others costs the host more or less with the size of the parameters. A serving layer (window queries,
// then this; 30 us a pass) against the 488 bytes of an older form, padded and timed in turn: 464 bytes +0.35 us, 472 and 480
// -0.1 to -0.3, 488 +0.2, 496 to 520 +0.3 to +0.45, 544 -0.2. What follows from other members is computed in the kernel.
static_assert(2 * sizeof(CUtensorMap) + sizeof(ResArgs) == 480, "kernel parameters");

// The head's chunk scores from the exchange into shared memory as order keys, two a word pair, as they arrive (src2: added); this thread's
// smallest and largest key. False: given up.
__device__ __forceinline__ bool take_scores(const ulonglong2* src, const ulonglong2* src2, int C, uint32_t tag, uint32_t* kbuf, uint32_t& lo,
                                            uint32_t& hi, volatile int* abort_flag) {
    constexpr int KP = 3;                // pairs in flight: one round trip up to 3456 chunks
    const int pairs = (C + 1) >> 1;
    for (int p0 = threadIdx.x; p0 < pairs; p0 += KP * kRThreads) {
        ulonglong2 a[KP], b[KP];
        unsigned missing = 0;
#pragma unroll
        for (int u = 0; u < KP; ++u) missing |= p0 + u * kRThreads < pairs ? 1u << u : 0u;
        const unsigned all = missing;
        long long t0 = 0;
        for (uint32_t it = 1;; ++it) {
#pragma unroll
            for (int u = 0; u < KP; ++u)
                if (missing >> u & 1u) {
                    a[u] = ld_tagged2(src + p0 + u * kRThreads);
                    if (src2 != nullptr) b[u] = ld_tagged2(src2 + p0 + u * kRThreads);
                }
#pragma unroll
            for (int u = 0; u < KP; ++u)
                if (missing >> u & 1u) {
                    const bool one = 2 * (p0 + u * kRThreads) + 1 == C;        // (no second chunk)
                    if (tagged_is(a[u].x, tag) && (one || tagged_is(a[u].y, tag)) &&
                        (src2 == nullptr || (tagged_is(b[u].x, tag) && (one || tagged_is(b[u].y, tag)))))
                        missing &= ~(1u << u);
                }
            if (missing == 0u) break;
            if ((it & 63u) == 0u) {
                if (t0 == 0) t0 = clock64();
                if (*abort_flag) return false;
                if (clock64() - t0 > kWaitLimitClocks) { *abort_flag = 1; return false; }
            }
        }
#pragma unroll
        for (int u = 0; u < KP; ++u)
            if (all >> u & 1u) {
                const int ch = 2 * (p0 + u * kRThreads);
                float x = tagged_value(a[u].x), y = tagged_value(a[u].y);
                if (src2 != nullptr) { x += tagged_value(b[u].x); y += tagged_value(b[u].y); }
                const uint32_t kx = select_order_key(x), ky = select_order_key(y);
                *reinterpret_cast<uint2*>(kbuf + ch) = make_uint2(kx, ky);
                lo = min(lo, kx);
                hi = max(hi, kx);
                if (ch + 1 < C) { lo = min(lo, ky); hi = max(hi, ky); }
            }
    }
    return true;
}
// The same from global memory, behind a hand-over by counters (rows padded to a multiple of four chunks).
__device__ __forceinline__ void load_scores(const float* sc, const float* sc2, int C, uint32_t* kbuf, uint32_t& lo, uint32_t& hi) {
    constexpr int KP = 4;
    const int pairs = (C + 1) >> 1;
    for (int p0 = threadIdx.x; p0 < pairs; p0 += KP * kRThreads) {
        float2 v[KP];
#pragma unroll
        for (int u = 0; u < KP; ++u) v[u] = __ldcg(reinterpret_cast<const float2*>(sc) + min(p0 + u * kRThreads, pairs - 1));
        if (sc2 != nullptr) {
#pragma unroll
            for (int u = 0; u < KP; ++u) {
                const float2 x = __ldcg(reinterpret_cast<const float2*>(sc2) + min(p0 + u * kRThreads, pairs - 1));
                v[u].x += x.x;
                v[u].y += x.y;
            }
        }
#pragma unroll
        for (int u = 0; u < KP; ++u) {
            const int ch = 2 * (p0 + u * kRThreads);
            if (ch < C) {
                const uint32_t kx = select_order_key(v[u].x), ky = select_order_key(v[u].y);
                *reinterpret_cast<uint2*>(kbuf + ch) = make_uint2(kx, ky);
                lo = min(lo, kx);
                hi = max(hi, kx);
                if (ch + 1 < C) { lo = min(lo, ky); hi = max(hi, ky); }
            }
        }
    }
}

// One thread publishes this CTA's arrival on `counter` and waits until `target` CTAs have arrived.
// Block-wide: every thread calls it; returns false if the wait was abandoned.
__device__ __forceinline__ bool head_handover(unsigned* counter, unsigned target, ResCtl& ctl) {
    __syncthreads();
    if (threadIdx.x == 0) {
        bool ok = true;
        // release: what this CTA wrote before the barrier above becomes visible to whoever acquires the count (and, behind
        // the barrier below, to the whole CTA); without a result the first poll follows at once
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
        const long long t0 = clock64();
        for (;;) {
            unsigned cur;
            asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(cur) : "l"(counter) : "memory");
            if (cur >= target) break;
            if (clock64() - t0 > kWaitLimitClocks) { ok = false; break; }
        }
        ctl.wait_ok = ok ? 1 : 0;
    }
    __syncthreads();
    return ctl.wait_ok != 0;
}

// BIG: two query tiles, or panels in scratch. A variant of its own: the code for either, present but not taken, costs
// the other shapes 1.5 us of 34 (32K tokens, 128 rows).
// FEW: up to 64 rows and more than kRManyCtas CTAs a head, for the reading of row statistics; a variant of its own for the same reason
// (as a run-time choice it costs every other shape 0.1 us of 12 to 30).
// WIDE: more than 16 chunks a thread (9216 a head), for the selection, whose bodies for them would slow the scoring of the others.
constexpr int kRManyCtas = 20;
template <int C_STATIC, bool BIG, bool FEW, bool WIDE>
__global__ void __launch_bounds__(kRThreads, 1)
layer_resident_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                      const ResArgs a) {
    constexpr int WP = panel_keys(C_STATIC);         // keys per epilogue panel
    constexpr int TILE = 2 * WP;                     // keys per accumulator tile
    constexpr uint32_t STAGE = TILE * 128;           // one ring stage: a tile's keys x 64 dims
    constexpr int SPP = WP / C_STATIC;               // chunk slots per panel
    constexpr uint32_t IDESC = umma_idesc_bf16(128, kRUmmaN);
    static_assert(WP % C_STATIC == 0, "the chunk size must divide the panel");

    extern __shared__ uint8_t smem_raw[];
    __shared__ ResCtl ctl;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int KB = a.d >> 6;
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* dyn = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t q_base = smem_base;
    const uint32_t k_base = smem_base + static_cast<uint32_t>(a.off_ring);
    float* pmax = reinterpret_cast<float*>(dyn + a.off_pmax);      // [panel of this CTA][128] panel maxima (log2 domain)
    float* misc = reinterpret_cast<float*>(dyn + a.off_misc);
    float* rec = misc;                 // [4 groups][{max, sum}][128]
    float* slice = misc + 1024;        // [4 slices][{max, sum}][128]; FEW: [{max, sum}][8 slices][64]
    float* gm = misc + 2048;           // [2 query tiles][128] row maxima of the head
    float* ginv = misc + 2304;         // [2 query tiles][128] 1 / row sums of the head
    uint8_t* ring = dyn + a.off_ring;  // reused after scoring
    volatile int* abort_flag = &ctl.abort_flag;
    const uint32_t n_stages = static_cast<uint32_t>(a.n_stages);

    const int hs = blockIdx.x / a.cph, part = blockIdx.x - hs * a.cph;      // scoring head, key range
    const int hkv = BIG ? hs : hs >> a.shift, row0 = BIG ? 0 : (hs & a.shift) * a.q_rows;
    const int n_rows = BIG ? a.R : (a.shift ? (row0 ? a.R - row0 : a.q_rows) : a.R);   // rows of the scoring head
    // tiles are dealt out rounding up, so the head's last CTA - whose last panels take the slow, masked path -
    // is never one of those that get an extra tile
    const int n_tiles = (a.L + TILE - 1) / TILE, C = (a.P + C_STATIC - 1) / C_STATIC;
    const int t_begin = (n_tiles * part + a.cph - 1) / a.cph, t_end = (n_tiles * (part + 1) + a.cph - 1) / a.cph;
    const int nt = t_end - t_begin;
    const int n_mt = BIG ? a.n_mt : 1;
    const bool two = n_mt == 2;                      // two query tiles
    const int n_vt = nt << (two ? 1 : 0);            // virtual tiles: (key tile, query tile) products of this CTA

    if (threadIdx.x == 0) {
        for (int s = 0; s < a.n_stages; ++s) {
            mbar_init(smem_u32(&ctl.full[s]), 1);
            mbar_init(smem_u32(&ctl.empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&ctl.tfull[b]), 1);
            mbar_init(smem_u32(&ctl.tempty[b]), 8);      // one arrival per warp of the pair that reads the buffer
        }
        mbar_init(smem_u32(&ctl.qfull), 1);
        for (int i = 0; i < 8; ++i) (&ctl.rec_count[0][0])[i] = 0;
        ctl.tag = 0u;
        ctl.abort_flag = 0;
        ctl.wait_ok = 1;
        prefetch_tmap(&tm_q);            // (kernel parameters: not written by the kernel ahead of this one)
        prefetch_tmap(&tm_k);
        fence_mbar_init();
        fence_proxy_async();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&ctl.tmem_base), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl.tmem_base;
    // Programmatic dependent launch (used when the launch asks for it, otherwise both are no-ops):
    // the next kernel of the stream may be set up while this one runs, and this one touches no
    // global memory before everything queued ahead of it has completed.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (elect_one() && nt > 0) {
            const uint32_t qbar = smem_u32(&ctl.qfull);
            mbar_arrive_expect_tx(qbar, static_cast<uint32_t>(n_mt * KB * a.q_rows) * 128u);
            for (int mt = 0; mt < n_mt; ++mt)      // (rows past R of the second tile arrive as zeros)
                for (int kb = 0; kb < KB; ++kb)
                    tma_load_3d(q_base + static_cast<uint32_t>(mt * KB + kb) * kRQTileBytes, &tm_q, qbar, kb * 64, row0 + mt * 128, hkv);
            const uint32_t k_bytes = static_cast<uint32_t>(min(a.L, TILE)) * 128u;
            // Panels in scratch: the keys leave the L2 to their records, unless the kept key rows, which the gather reads again, are
            // many. us without -> with the hint (kept key rows): 131072 tokens, 256 rows, c = 20 (8 MB) 124 -> 115; 131072, 128 rows, c = 10 (13 MB) 85.2 -> 82.5;
            // 52088, 64 rows, c = 5 (17 MB) 55.7 -> 54.0; 80000, 128 rows, c = 10 (25 MB) 64.4 -> 63.2; 120859, 128 rows, c = 20 (45 MB) 92.4 -> 98.3; 131072,
            // 64 rows, c = 5 (67 MB) 146.7 -> 149.2.
            const bool keys_leave = a.n_off > 0 && 2ll * a.n_max * a.Hkv * a.d <= (32ll << 20);
            const uint64_t policy = keys_leave ? l2_policy_evict_first() : l2_policy_evict_normal();
            uint32_t st = 0, st_par = 1;
            int issued = 0;
            bool ok = true;
            for (int t = t_begin; t < t_end && ok; ++t) {
                for (int kb = 0; kb < KB; ++kb) {
                    ok = mbar_wait(smem_u32(&ctl.empty[st]), st_par, abort_flag);
                    if (!ok) break;
                    const uint32_t bar = smem_u32(&ctl.full[st]);
                    mbar_arrive_expect_tx(bar, k_bytes);
                    if constexpr (BIG) tma_load_3d_hint(k_base + st * STAGE, &tm_k, bar, kb * 64, t * TILE, hkv, policy);
                    else tma_load_3d(k_base + st * STAGE, &tm_k, bar, kb * 64, t * TILE, hkv);
                    ++issued;
                    if (++st == n_stages) { st = 0; st_par ^= 1u; }
                }
            }
            if (!ok) {
                // Give copies already in flight a bounded chance to land before the CTA exits.
                const int back = min(issued, a.n_stages);
                for (int i = 1; i <= back; ++i) {
                    const int cc = issued - i, s = cc % a.n_stages;
                    const long long t0 = clock64();
                    while (!mbar_try_wait(smem_u32(&ctl.full[s]), (cc / a.n_stages) & 1) &&
                           clock64() - t0 < kWaitLimitClocks / 8) {
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ UMMA issuer
        if (elect_one() && nt > 0) {
            bool ok = mbar_wait(smem_u32(&ctl.qfull), 0, abort_flag);
            const uint64_t q_desc = umma_desc_sw128(q_base), k_desc = umma_desc_sw128(k_base);
            const bool both = KB == 2;                   // d is 64 or 128: one or two stages a tile
            uint32_t st = 0, st_par = 0;
            for (int ti = 0, vt = 0; ti < nt && ok; ++ti) {
                const uint32_t s0 = st, p0 = st_par;
                if (++st == n_stages) { st = 0; st_par ^= 1u; }
                const uint32_t s1 = both ? st : s0, p1 = both ? st_par : p0;
                if (both && ++st == n_stages) { st = 0; st_par ^= 1u; }
                for (int mt = 0; mt < n_mt; ++mt, ++vt) {
                    const int buf = vt & 1, use = vt >> 1;
                    const uint32_t tempty = smem_u32(&ctl.tempty[buf]), te_par = (use & 1) ^ 1;
                    ok = mt == 0 ? mbar_wait3(smem_u32(&ctl.full[s0]), p0, smem_u32(&ctl.full[s1]), p1, tempty, te_par, abort_flag)
                                 : mbar_wait(tempty, te_par, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    issue_products(tmem_base + static_cast<uint32_t>(buf * kRUmmaN), q_desc + static_cast<uint32_t>(mt * KB) * (kRQTileBytes >> 4),
                                   k_desc + s0 * (STAGE >> 4), k_desc + s1 * (STAGE >> 4), both, IDESC);
                    umma_commit(smem_u32(&ctl.tfull[buf]));
                }
                if (!ok) break;
                umma_commit(smem_u32(&ctl.empty[s0]));
                if (both) umma_commit(smem_u32(&ctl.empty[s1]));
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        // Four groups of four warps (a group's warps cover the four tensor-memory lane quarters =
        // 128 query rows). The groups form two pairs that take alternate virtual tiles; inside a
        // pair each group takes one half (panel) of the tile.
        const int grp = (warp - 2) >> 2, quarter = warp & 3;
        const int pair = grp >> 1, half = grp & 1;
        const int row = quarter * 32 + lane;             // row of the query tile = lane of tensor memory
        const int qrow = row + (two ? pair * 128 : 0);   // row of the KV head
        const bool active = qrow < n_rows;
        const int last_visible = a.P + ((row0 + qrow) % a.w);     // this row sees keys j <= P + r (all < L)
        const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        const uint64_t keep = l2_policy_evict_last();
        // (behind griddepcontrol.wait; beside the first keys' way here, which the issuing thread should not wait for twice)
        if (a.direct != 0 && threadIdx.x == 64) *const_cast<volatile uint32_t*>(&ctl.tag) = take_tag(*a.x);
        float run_m = -CUDART_INF_F, run_l = 0.f;
        bool scored = true;
        for (int vt = pair; vt < n_vt; vt += 2) {
            const int use = vt >> 1, ti = two ? use : vt;
            scored = mbar_wait_warp(smem_u32(&ctl.tfull[pair]), use & 1, abort_flag);
            if (!scored) break;
            tc_fence_after();
            float v[WP];
            load_panel<WP>(lane_addr + static_cast<uint32_t>(pair * kRUmmaN + half * WP), v);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl.tempty[pair]));   // the buffer may be overwritten now
            const int pl = vt * 2 + half;                // panel of this CTA; pl % 4 == grp
            const int j0 = (t_begin + ti) * TILE + half * WP;
            float pr[SPP], m2, l;
            auto emit = [&](int ch, float acc) { pr[ch] = acc; };
            if (j0 + WP <= a.P)
                panel_fast<C_STATIC, WP>(v, a.sl2, emit, &m2, &l);
            else
                panel_static_tail<C_STATIC, WP>(v, a.sl2, emit, j0, a.P, last_visible, &m2, &l);
            if (!BIG || pl < a.n_on) {
                part_store<SPP>(lane_addr + static_cast<uint32_t>(kRPartCol0 + pl * SPP), pr);
                pmax[pl * 128 + row] = m2;
            } else {
                float rec_[SPP + 1];
#pragma unroll
                for (int q = 0; q < SPP; ++q) rec_[q] = pr[q];
                rec_[SPP] = m2;
                const size_t at = static_cast<size_t>(blockIdx.x) * a.n_off + (pl - a.n_on);
                if (a.spill_rows == 128)
                    spill_store<SPP + 1, 128>(a.spill + at * ((SPP + 1) * 128), 128, row, rec_, keep);
                else if (active)
                    spill_store<SPP + 1, 0>(a.spill + at * ((SPP + 1) * a.spill_rows), a.spill_rows, row, rec_, keep);
            }
            // the running record: l is relative to m2, run_l to run_m
            merge_ml(run_m, run_l, m2, l);
        }
        tmem_st_wait();
        rec[(grp * 2 + 0) * 128 + row] = active ? run_m : -CUDART_INF_F;
        rec[(grp * 2 + 1) * 128 + row] = active ? run_l : 0.f;

        // ---- 2. (hand-over that carries its data) The last of the warps that hold the same 32 rows merges their parts and stores them; then
        // every thread takes its share of the records of one row of the head: a slice a group, the slices are put together below.
        // Up to 64 rows and more CTAs a head than four slices of records read in one round trip (2 heads: 74): eight slices of 64 rows.
        if (a.direct != 0 && scored) {
            __threadfence_block();
            __syncwarp();
            const int mt = two ? pair : 0, n_g = two ? 2 : 4;
            const uint32_t tag = wait_tag(&ctl.tag, abort_flag);
            int old = 0;
            if (lane == 0) old = atomicAdd(&ctl.rec_count[mt][quarter], 1);
            if (__shfl_sync(0xffffffffu, old, 0) == n_g - 1) {
                __threadfence_block();
                float M = -CUDART_INF_F, S = 0.f, m[4], l[4];
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    m[g] = g < n_g ? rec[((mt * 2 + g) * 2) * 128 + row] : -CUDART_INF_F;
                    l[g] = g < n_g ? rec[((mt * 2 + g) * 2 + 1) * 128 + row] : 0.f;
                }
                merge_records(M, S, m, l);
                if (tag != 0u) st_tagged2(&a.x->record[(static_cast<size_t>(blockIdx.x) * n_mt + mt) * 128 + row], M, S, tag);
            }
            constexpr int KF = BIG ? 9 : 5;              // records in flight per thread: one round trip where a head has 18 CTAs (8 heads)
            const int n_sl = FEW ? 8 : (two ? 2 : 4), sl = FEW ? grp * 2 + (quarter >> 1) : (two ? half : grp);
            const int prow = FEW ? (quarter & 1) * 32 + lane : row;
            float M = -CUDART_INF_F, S = 0.f;
            if (tag != 0u && (FEW ? prow < n_rows : active)) {
                const size_t step = static_cast<size_t>(n_mt) * 128;
                const ulonglong2* src = a.x->record + (static_cast<size_t>(hs) * a.cph * n_mt + mt) * 128 + prow;
                for (int j0 = sl; j0 < a.cph; j0 += KF * n_sl)
                    if (!take_records<KF, FEW>(src + j0 * step, n_sl * step, min(KF, (a.cph - j0 + n_sl - 1) / n_sl), tag, M, S, abort_flag)) break;
            }
            if constexpr (FEW) {
                slice[sl * 64 + prow] = M;
                slice[512 + sl * 64 + prow] = S;
            } else {
                slice[(grp * 2 + 0) * 128 + row] = M;
                slice[(grp * 2 + 1) * 128 + row] = S;
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    bool ok = ctl.abort_flag == 0;

    // ---- 2. (by counters) this CTA's (max, sum) per row -> global memory; wait for the head's other CTAs
    if (ok && a.direct == 0) {
        if (static_cast<int>(threadIdx.x) < n_mt * 128) {
            const int i = threadIdx.x & 127;
            const int g0 = two ? (threadIdx.x >> 7) * 2 : 0, g1 = two ? g0 + 2 : 4;   // groups that scored this query tile
            float M = -CUDART_INF_F, Ls = 0.f;
#pragma unroll
            for (int g = 0; g < 4; ++g)
                if (g >= g0 && g < g1) M = fmaxf(M, rec[(g * 2) * 128 + i]);
#pragma unroll
            for (int g = 0; g < 4; ++g)
                if (g >= g0 && g < g1) {
                    const float m = rec[(g * 2) * 128 + i];
                    Ls += rec[(g * 2 + 1) * 128 + i] * ex2_below(m, M);
                }
            float* dst = a.cta_stat + (static_cast<size_t>(blockIdx.x) * n_mt + (threadIdx.x >> 7)) * 256;
            dst[i] = M;
            dst[128 + i] = Ls;
        }
        ok = head_handover(a.cnt_a(hs), static_cast<unsigned>(a.cph), ctl);
    }

    // ---- 3. row statistics of the head, then this CTA's chunk scores
    if (ok) {
        if (a.direct == 0) {
            if constexpr (FEW) {
                float M = -CUDART_INF_F, Ls = 0.f;
                if (threadIdx.x < 512) {
                    const float* src = a.cta_stat + static_cast<size_t>(hs) * a.cph * 256 + (threadIdx.x & 63);
#pragma unroll 1
                    for (int j0 = threadIdx.x >> 6; j0 < a.cph; j0 += 40) {
                        float rm[5], rl[5];
#pragma unroll
                        for (int u = 0; u < 5; ++u) {
                            const int j = j0 + 8 * u;
                            rm[u] = (j < a.cph) ? __ldcg(src + j * 256) : -CUDART_INF_F;
                            rl[u] = (j < a.cph) ? __ldcg(src + j * 256 + 128) : 0.f;
                        }
#pragma unroll
                        for (int u = 0; u < 5; ++u) merge_ml(M, Ls, rm[u], rl[u]);
                    }
                    slice[threadIdx.x] = M;
                    slice[512 + threadIdx.x] = Ls;
                }
                __syncthreads();
                if (threadIdx.x < 64) {
#pragma unroll
                    for (int s = 1; s < 8; ++s) merge_ml(M, Ls, slice[s * 64 + threadIdx.x], slice[512 + s * 64 + threadIdx.x]);
                    gm[threadIdx.x] = M;
                    ginv[threadIdx.x] = 1.0f / Ls;
                }
            }
            // 512 threads: four (one query tile) or two (two tiles) slices of the records per row
            if constexpr (!FEW) {
                const int n_sl = two ? 2 : 4;
                if (threadIdx.x < 512) {
                    const int i = threadIdx.x & 127, sl = (threadIdx.x >> 7) & (n_sl - 1), mt = two ? threadIdx.x >> 8 : 0;
                    const size_t step = static_cast<size_t>(n_mt) * 256;
                    const float* src = a.cta_stat + (static_cast<size_t>(hs) * a.cph * n_mt + mt) * 256 + i;
                    float M = -CUDART_INF_F, Ls = 0.f;
                    // records in flight per thread: enough for one round trip where a head has 18 CTAs (8 heads)
                    constexpr int kF = BIG ? 9 : 5;
                    for (int j0 = sl; j0 < a.cph; j0 += kF * n_sl) {
                        float rm[kF], rl[kF];
#pragma unroll
                        for (int u = 0; u < kF; ++u) {
                            const int j = j0 + n_sl * u;
                            rm[u] = (j < a.cph) ? __ldcg(src + j * step) : -CUDART_INF_F;
                            rl[u] = (j < a.cph) ? __ldcg(src + j * step + 128) : 0.f;
                        }
                        float bm = M;
#pragma unroll
                        for (int u = 0; u < kF; ++u) bm = fmaxf(bm, rm[u]);
                        float acc = Ls * ex2_below(M, bm);
#pragma unroll
                        for (int u = 0; u < kF; ++u) acc += rl[u] * ex2_below(rm[u], bm);
                        M = bm;
                        Ls = acc;
                    }
                    slice[((threadIdx.x >> 7) * 2 + 0) * 128 + i] = M;
                    slice[((threadIdx.x >> 7) * 2 + 1) * 128 + i] = Ls;
                }
                __syncthreads();
                if (static_cast<int>(threadIdx.x) < n_mt * 128) {
                    const int i = threadIdx.x & 127, s0 = (threadIdx.x >> 7) * n_sl;
                    float M = -CUDART_INF_F, Ls = 0.f;
#pragma unroll
                    for (int s = 0; s < 4; ++s)
                        if (s >= s0 && s < s0 + n_sl) M = fmaxf(M, slice[(s * 2) * 128 + i]);
#pragma unroll
                    for (int s = 0; s < 4; ++s)
                        if (s >= s0 && s < s0 + n_sl) {
                            const float m = slice[(s * 2) * 128 + i];
                            Ls += slice[(s * 2 + 1) * 128 + i] * ex2_below(m, M);
                        }
                    gm[threadIdx.x] = M;
                    ginv[threadIdx.x] = 1.0f / Ls;       // rows >= R are never used
                }
            }
            __syncthreads();
        }
        // chunk scores of this CTA's key range: partial sums x exp2(m_panel - m_i) / l_i, summed over
        // the rows. A thread holds one row of up to 32 chunk slots at a time (PPB panels of its
        // group: panels grp, grp + 4, ...); a transposing warp reduction leaves lane j with the sum
        // over the warp's 32 rows of slot j; the lane quarters (and query tiles) are added through
        // shared memory (the K ring is idle now).
        float* red = reinterpret_cast<float*>(ring);     // [query tiles x 4 lane quarters][chunk slots of this CTA]
        const int n_local = nt * (TILE / C_STATIC);      // chunk slots of this CTA
        const int n_pl = 2 * n_vt;
        if (warp >= 2) {
            const int grp = (warp - 2) >> 2, quarter = warp & 3;
            const int row = quarter * 32 + lane, mt = two ? grp >> 1 : 0;
            const bool active = mt * 128 + row < n_rows;
            const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
            const int srow = active ? row : 0;           // (rows that do not exist have no record)
            float mi, li;                                // the row's maximum and 1 / sum in the head (rows >= R: never used)
            if (a.direct == 0) {
                mi = gm[mt * 128 + row];
                li = ginv[mt * 128 + row];
            } else {
                float M = -CUDART_INF_F, S = 0.f;
                if constexpr (FEW) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) merge_ml(M, S, slice[u * 64 + (row & 63)], slice[512 + u * 64 + (row & 63)]);
                } else {
                    float m[4], l[4];
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        const bool mine = !two || (g >> 1) == mt;
                        m[g] = mine ? slice[(g * 2) * 128 + row] : -CUDART_INF_F;
                        l[g] = mine ? slice[(g * 2 + 1) * 128 + row] : 0.f;
                    }
                    merge_records(M, S, m, l);
                }
                mi = M;
                li = 1.0f / S;
            }
            const uint64_t drop = l2_policy_evict_first();   // the sums in scratch are dead once read
            constexpr int PPB = 32 / SPP;                // panels per block of up to 32 values
            for (int b0 = 0; grp + 4 * b0 < n_pl; b0 += PPB) {
                float v[32], pm[PPB];
                // (panel numbers clamped: every lane issues the same loads) A block that is on chip as a whole - every
                // block of most shapes - takes its loads without a branch between them, so that they overlap.
                if (!BIG || min(grp + 4 * (b0 + PPB - 1), n_pl - 1) < a.n_on) {
#pragma unroll
                    for (int u = 0; u < PPB; ++u) {
                        const int pl = min(grp + 4 * (b0 + u), n_pl - 1);
                        part_load<SPP>(lane_addr + static_cast<uint32_t>(kRPartCol0 + pl * SPP), &v[u * SPP]);
                        pm[u] = pmax[pl * 128 + row];
                    }
                } else {
#pragma unroll
                    for (int u = 0; u < PPB; ++u) {
                        const int pl = min(grp + 4 * (b0 + u), n_pl - 1);
                        if (pl < a.n_on) {
                            part_load<SPP>(lane_addr + static_cast<uint32_t>(kRPartCol0 + pl * SPP), &v[u * SPP]);
                            pm[u] = pmax[pl * 128 + row];
                        } else {
                            float rec_[SPP + 1];
                            const size_t at = static_cast<size_t>(blockIdx.x) * a.n_off + (pl - a.n_on);
                            if (a.spill_rows == 128)
                                spill_load<SPP + 1, 128>(a.spill + at * ((SPP + 1) * 128), 128, row, rec_, drop);
                            else
                                spill_load<SPP + 1, 0>(a.spill + at * ((SPP + 1) * a.spill_rows), a.spill_rows, srow, rec_, drop);
                            pm[u] = rec_[SPP];
#pragma unroll
                            for (int q = 0; q < SPP; ++q) v[u * SPP + q] = rec_[q];
                        }
                    }
                }
                tmem_ld_wait();
#pragma unroll
                for (int e = PPB * SPP; e < 32; ++e) v[e] = 0.f;
#pragma unroll
                for (int u = 0; u < PPB; ++u) {
                    const bool have = active && grp + 4 * (b0 + u) < n_pl;
                    const float f = have ? ex2_approx(pm[u] - mi) * li : 0.f;
#pragma unroll
                    for (int s = 0; s < SPP; ++s) v[u * SPP + s] = have ? v[u * SPP + s] * f : 0.f;
                }
                const float tot = warp_transpose_reduce(v, lane);
                const int pl = grp + 4 * (b0 + lane / SPP);
                if (lane < PPB * SPP && pl < n_pl) {
                    const int kp = two ? (pl >> 2) * 2 + (pl & 1) : pl;      // panel of the key range
                    red[(mt * 4 + quarter) * n_local + kp * SPP + lane % SPP] = tot;
                }
            }
        }
        tc_fence_before();
        __syncthreads();
        const int ch0 = t_begin * (TILE / C_STATIC);     // this CTA's first chunk
        for (int lc = threadIdx.x; lc < n_local; lc += kRThreads)
            if (ch0 + lc < C) {
                const float* r = red + lc;
                float t = (r[0] + r[n_local]) + (r[2 * n_local] + r[3 * n_local]);
                if (two) t += (r[4 * n_local] + r[5 * n_local]) + (r[6 * n_local] + r[7 * n_local]);
                const size_t at = static_cast<size_t>(hs) * a.score_row + ch0 + lc;
                if (a.direct & kDirectScores) st_tagged(reinterpret_cast<unsigned long long*>(a.x->score) + at, t, ctl.tag);
                else a.scores[at] = t;
            }
    }
    // ---- 4. wait for the KV head's other CTAs, 5. select, 6. gather
    if (ok && a.out_idx != nullptr) {
        if (a.direct & kDirectScores) __syncthreads();       // (the sums above are read; the ring is written again)
        else ok = head_handover(a.cnt_b(hkv), static_cast<unsigned>(a.cph << (BIG ? 0 : a.shift)), ctl);
    }
    if (ok && a.out_idx != nullptr) {
        SelectSmem& ss = *reinterpret_cast<SelectSmem*>(ring);
        const int shift = BIG ? 0 : a.shift;
        const size_t row_at = (static_cast<size_t>(hkv) << shift) * a.score_row;
        const float* sc = a.scores + row_at;
        const float* sc2 = shift ? sc + a.score_row : nullptr;           // the other half's chunk scores are added
        const int Q = a.cph << shift, q = (hs & shift) * a.cph + part;   // CTAs of this KV head
        const int r_begin = static_cast<int>(static_cast<long long>(a.n_max) * q / Q);
        const int r_end = static_cast<int>(static_cast<long long>(a.n_max) * (q + 1) / Q);
        int32_t* out_idx = a.out_idx + static_cast<size_t>(hkv) * a.n_max;
        uint32_t* kbuf = reinterpret_cast<uint32_t*>(ring + kRSelBytes);
        // every CTA holds the head's kept chunks: it expands, writes and gathers its own share of the positions
        const bool listed = lists_kept(WIDE, C, a.k, a.ring_bytes);
        if constexpr (WIDE) {
            if (listed) select_kept<kSelLayerWide>(sc, sc2, C, a.k, ss, kbuf);
        } else {
            if (listed && !select_all(C, a.k, ss)) {
                uint32_t lo = 0xffffffffu, hi = 0u;
                select_clear(ss);
                if (a.direct & kDirectScores) {
                    const ulonglong2* x = a.x->score + row_at / 2;
                    take_scores(x, shift ? x + a.score_row / 2 : nullptr, C, ctl.tag, kbuf, lo, hi, abort_flag);
                } else {
                    load_scores(sc, sc2, C, kbuf, lo, hi);
                }
                lo = __reduce_min_sync(0xffffffffu, lo);
                hi = __reduce_max_sync(0xffffffffu, hi);
                if (lane == 0) ss.warp_sums[warp] = (static_cast<unsigned long long>(hi) << 32) | lo;
                __syncthreads();
                ok = ctl.abort_flag == 0;
                if (ok) {
                    const int per = (C + kRThreads - 1) / kRThreads;
                    // (runs of 6 and 12 as well: 3274 chunks 28.94 -> 28.59 us a layer, 6550 20.98 -> 20.65)
                    if (per <= 2) select_staged<2>(kbuf, C, a.k, ss);
                    else if (per <= 4) select_staged<4>(kbuf, C, a.k, ss);
                    else if (per <= 6) select_staged<6>(kbuf, C, a.k, ss);
                    else if (per <= 8) select_staged<8>(kbuf, C, a.k, ss);
                    else if (per <= 12) select_staged<12>(kbuf, C, a.k, ss);
                    else select_staged<16>(kbuf, C, a.k, ss);
                }
            }
        }
        // very many chunks, or very many kept: every CTA of the head writes the same positions to out_idx and takes its share from there
        if (!listed) {
            select_head_rows(sc, sc2, a.L, a.w, C_STATIC, C, a.k, a.n_max, out_idx, ss, keys_fit(C, a.ring_bytes) ? kbuf : nullptr, a.tok_cap);
            __syncthreads();
        }
        if (ok) {
            const int n_tok = listed ? select_tokens(a.P, C_STATIC, C, a.k, ss, a.tok_cap) : 0;
            auto index_at = [&](int n) { return listed ? select_position(ss, n, n_tok, C_STATIC, a.P, a.w) : __ldcg(out_idx + n); };
            int32_t* idx_out = listed ? out_idx : nullptr;
            const int vpr = a.d >> 3;
            const int rows_per_pass = (kRThreads / vpr) * kGatherRowsPerThread;
            // packed outputs: this head's block; paged outputs: the cache base (rows are placed through the block table)
            const PagedDst pg{a.block_table, a.page_size, a.num_pages, a.Hkv, hkv};
            const size_t head_out = a.block_table ? 0 : static_cast<size_t>(hkv) * a.n_max;
            const uint4* Kh = a.K + static_cast<size_t>(hkv) * a.k_head;
            const uint4* Vh = a.V + static_cast<size_t>(hkv) * a.v_head;
            for (int n0 = r_begin; n0 < r_end; n0 += rows_per_pass) {
                if (vpr == 16)
                    gather_rows_at<16>(Kh, Vh, index_at, a.L, r_end, n0, threadIdx.x, kRThreads, a.out_K + head_out * 16, a.out_V + head_out * 16,
                                       idx_out, a.k_row, a.v_row, pg);
                else
                    gather_rows_at<8>(Kh, Vh, index_at, a.L, r_end, n0, threadIdx.x, kRThreads, a.out_K + head_out * 8, a.out_V + head_out * 8,
                                      idx_out, a.k_row, a.v_row, pg);
            }
        }
    }
    // tensor memory has not been read since the barrier after the contraction (or after scoring)
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    if (threadIdx.x == 0) {
        if (!ok) atomicExch(a.status(), 1);
        // The last CTA to leave clears the hand-over counters for the next launch, if there were any. (After an
        // abandoned wait the counters are left as they are; chunkkv_device_status clears them.)
        const bool counted = a.direct == 0 || (a.direct == kDirectRecords && a.out_idx != nullptr);
        const bool last_tag = a.direct != 0 && ctl.tag == kLastTag;
        if ((counted || last_tag) && atomicAdd(a.exits(), 1u) + 1u == gridDim.x) {
            for (int h = 0; h < a.Hkv << a.shift; ++h) { *a.cnt_a(h) = 0u; *a.cnt_b(h) = 0u; }
            *a.exits() = 0u;
            if (last_tag) end_tags(*a.x);
            __threadfence();
        }
    }
}

// variant: 0 small, 1 big, 2 small with few rows
template <int C_STATIC, bool WIDE>
const void* kernel_of(int variant) {
    return variant == 1 ? reinterpret_cast<const void*>(layer_resident_kernel<C_STATIC, true, false, WIDE>)
         : variant == 2 ? reinterpret_cast<const void*>(layer_resident_kernel<C_STATIC, false, true, WIDE>)
                        : reinterpret_cast<const void*>(layer_resident_kernel<C_STATIC, false, false, WIDE>);
}

template <int C_STATIC>
const void* kernel_of(int variant, bool wide) {
    return wide ? kernel_of<C_STATIC, true>(variant) : kernel_of<C_STATIC, false>(variant);
}

}  // namespace

cudaError_t exchange_slots(Exchange** slots) { return cudaGetSymbolAddress(reinterpret_cast<void**>(slots), g_exchange); }
Exchange* exchange_slot(Exchange* slots, int slot) { return slots + slot; }
uint32_t* exchange_tags(Exchange* x) { return &x->last_tag; }

size_t resident_scratch_floats(const ResidentPlan& plan, int Hkv, int C) {
    return static_cast<size_t>(plan.grid) * plan.n_mt * 256 + (((static_cast<size_t>(Hkv) << plan.shift) * ((C + 3) & ~3) + 63) & ~static_cast<size_t>(63)) +
           static_cast<size_t>(plan.grid) * plan.n_off * (plan.spp + 1) * plan.spill_rows;
}

bool make_resident_plan(int L, int R, int Hkv, int d, int c, int C, int n_max, int max_ctas, int smem_limit,
                        ResidentPlan* plan) {
    // The chunk sizes that are compiled in: of those that divide a panel of 60 or 64 keys, 5, 10 and 20 of the method's
    // ablation and the page sizes 8, 16 and 32. 3, 4, 6, 12, 15 and 30 divide 60 as well and would fit; each costs two
    // kernels here, two in model_kernel.cu and 3 MB of library. They and the sizes that divide neither take the kernels of
    // score.cu (32768 tokens, 128 rows: c = 15 88 us, c = 16 here 29), token level token_kernel.cu.
    if (c != 5 && c != 8 && c != 10 && c != 16 && c != 20 && c != 32) return false;
    if (R < 1 || R > 256 || (d != 64 && d != 128) || L < 1 || C < 1 || Hkv < 1 || Hkv > kResidentMaxHeads) return false;
    if (max_ctas < Hkv) return false;
    ResidentPlan p{};
    p.c_static = c;
    const int tile = 2 * panel_keys(c);
    p.spp = panel_keys(c) / c;
    p.tile = tile;
    p.n_tiles = (L + tile - 1) / tile;
    // More than 128 rows as two scoring heads where all panels of such a head stay on chip (see the top of this file); chunk
    // scores alone (no positions to fill) always as two query tiles, which leave nothing to add afterwards.
    const int halves = max_ctas / (2 * Hkv) < p.n_tiles ? max_ctas / (2 * Hkv) : p.n_tiles;
    if (R > 128 && n_max > 0 && halves > 0 && 2 * Hkv <= kResidentMaxHeads) {
        const int t = (p.n_tiles + halves - 1) / halves;
        p.shift = 2 * t * p.spp <= kRPartCols ? 1 : 0;
    }
    p.n_mt = R > 128 && p.shift == 0 ? 2 : 1;
    p.cph = max_ctas / (Hkv << p.shift);
    if (p.cph > p.n_tiles) p.cph = p.n_tiles;                       // a CTA without keys would only lengthen the hand-overs
    p.grid = p.cph * (Hkv << p.shift);
    p.t_max = (p.n_tiles + p.cph - 1) / p.cph;
    const int n_pl = 2 * p.n_mt * p.t_max;                          // panels of a CTA
    p.n_on = kRPartCols / p.spp;
    if (p.n_on > n_pl) p.n_on = n_pl;
    p.n_off = n_pl - p.n_on;
    p.spill_rows = R < 128 ? (R + 3) & ~3 : 128;                    // 16-byte aligned records of the rows that exist
    const int KB = d / 64, stage = tile * 128;
    const int q_bytes = p.n_mt * KB * kRQTileBytes;
    const int pmax_bytes = p.n_on * 128 * 4;
    const int fixed = 1024 /* alignment */ + q_bytes + 1024 /* tail of the last stage's UMMA read */ + pmax_bytes + kRMiscBytes;
    int ns = (smem_limit - fixed) / stage;
    if (ns > kRMaxStages) ns = kRMaxStages;
    if (ns < 2 * KB) return false;
    p.n_stages = ns;
    p.off_ring = q_bytes;
    p.ring_bytes = ns * stage + 1024;
    p.off_pmax = p.off_ring + p.ring_bytes;
    p.off_misc = p.off_pmax + pmax_bytes;
    p.smem_bytes = 1024 + p.off_misc + kRMiscBytes;
    // After scoring the ring holds the row sums of the chunk scores, then the selection's scratch and keys. (A CTA's kept positions, which it
    // once held as well, still have to have room: calls with more of them stay with the kernels of score.cu.)
    if (static_cast<size_t>(p.n_mt) * 4 * p.t_max * (tile / c) * 4 > static_cast<size_t>(p.ring_bytes)) return false;
    const size_t own = static_cast<size_t>(n_max) / (p.cph << p.shift) + 1;      // kept positions of a CTA
    const size_t sel_bytes = ((sizeof(SelectSmem) + 127) & ~size_t(127)) + ((own * 4 + 127) & ~size_t(127));
    if (sel_bytes > static_cast<size_t>(p.ring_bytes)) return false;
    *plan = p;
    return true;
}

cudaError_t launch_layer_resident(const ResidentPlan& plan, const CUtensorMap& tm_q, const CUtensorMap& tm_k,
                                  const ResidentIO& io, cudaStream_t stream) {
    const bool wide = io.out_idx != nullptr && io.C > kRThreads * select_reg_keys(kSelLayer);
    ResArgs a{};
    a.L = io.L; a.P = io.L - io.w; a.w = io.w; a.R = io.R; a.d = io.d; a.n_mt = static_cast<short>(plan.n_mt);
    a.sl2 = io.sl2;
    a.cph = plan.cph; a.n_stages = plan.n_stages;
    a.direct = io.cooperative || io.exchange == nullptr || !resident_tagged(plan) ? 0
             : kDirectRecords | (io.out_idx != nullptr && !wide && lists_kept(false, io.C, io.k, plan.ring_bytes) &&
                               static_cast<long long>(io.Hkv << plan.shift) * ((io.C + 3) & ~3) <= kXScores ? kDirectScores : 0);
    a.shift = static_cast<short>(plan.shift); a.q_rows = resident_q_box_rows(plan, io.R);
    a.k = io.k; a.n_max = io.n_max; a.Hkv = io.Hkv;
    a.n_on = plan.n_on; a.n_off = plan.n_off; a.spill_rows = plan.spill_rows;
    a.off_ring = plan.off_ring; a.ring_bytes = plan.ring_bytes; a.off_pmax = plan.off_pmax; a.off_misc = plan.off_misc;
    a.K = static_cast<const uint4*>(io.K); a.V = static_cast<const uint4*>(io.V);
    a.block_table = io.block_table; a.page_size = io.page_size; a.num_pages = io.num_pages;
    a.tok_cap = io.tok_cap;
    {
        const long long vpr = io.d / 8;
        a.k_row = io.k_row_elems ? io.k_row_elems / 8 : vpr;
        a.v_row = io.v_row_elems ? io.v_row_elems / 8 : vpr;
        a.k_head = io.k_head_elems ? io.k_head_elems / 8 : static_cast<long long>(io.L) * vpr;
        a.v_head = io.v_head_elems ? io.v_head_elems / 8 : static_cast<long long>(io.L) * vpr;
    }
    a.out_K = static_cast<uint4*>(io.out_K); a.out_V = static_cast<uint4*>(io.out_V); a.out_idx = io.out_idx;
    if (a.direct != 0) a.x = io.exchange;
    else a.cta_stat = io.scratch;
    float* scores = io.scratch + static_cast<size_t>(plan.grid) * plan.n_mt * 256;
    a.scores = io.out_scores ? io.out_scores : scores;
    a.score_row = io.out_scores ? io.C : (io.C + 3) & ~3;
    a.spill = scores + (((static_cast<size_t>(io.Hkv) << plan.shift) * ((io.C + 3) & ~3) + 63) & ~static_cast<size_t>(63));
    a.counters = io.counters;
    const int variant = plan.n_mt == 2 || plan.n_off > 0 ? 1 : (io.R <= 64 && plan.cph > kRManyCtas ? 2 : 0);
    const void* kern = nullptr;
    int v = 0;
    switch (plan.c_static) {
        case 5: kern = kernel_of<5>(variant, wide); v = 0; break;
        case 8: kern = kernel_of<8>(variant, wide); v = 1; break;
        case 10: kern = kernel_of<10>(variant, wide); v = 2; break;
        case 16: kern = kernel_of<16>(variant, wide); v = 3; break;
        case 20: kern = kernel_of<20>(variant, wide); v = 4; break;
        case 32: kern = kernel_of<32>(variant, wide); v = 5; break;
        default: return cudaErrorInvalidValue;
    }
    v += 6 * (variant + (wide ? 3 : 0));
    static int smem_set[36][64] = {{0}};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || smem_set[v][dev] < plan.smem_bytes) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, plan.smem_bytes);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) smem_set[v][dev] = plan.smem_bytes;
    }
    void* params[] = {const_cast<CUtensorMap*>(&tm_q), const_cast<CUtensorMap*>(&tm_k), &a};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(plan.grid);
    cfg.blockDim = dim3(kRThreads);
    cfg.dynamicSmemBytes = static_cast<size_t>(plan.smem_bytes);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    if (io.cooperative) {
        // several such launches may share the GPU (lanes): each must have all of its CTAs resident
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    } else {
        // One launch at a time on the device (the calls share one scratch buffer and are ordered): at
        // most one CTA per SM and no more CTAs than SMs, so every CTA becomes resident without
        // waiting for another CTA of this grid. Launched as a programmatic dependent of the
        // preceding kernel, the set-up of this one overlaps the end of that one.
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, kern, params);
}

}  // namespace chunkkv
