// Token scores (ChunkKV Algorithm 3 with chunk size 1, the token-level selection of the paper's
// hybrid experiment; also chunkkv_score's token-score output): t[j] = sum over the window rows of
// softmax(q k^T / sqrt(d))[i, j] for every prefix key j.
//
// With one chunk per key the per-(chunk, row) partial sums of the other kernels would be the whole
// score matrix, so this kernel walks its keys twice instead, in one launch: pass 1 only folds the
// per-row (max, sum) of the CTA's key range; the CTAs of a head exchange those records (words
// that carry the launch's tag, bounded waits); pass 2 recomputes the same tiles (the keys come back from L2),
// normalises every element with the final row statistics and sums over the rows. Pass 1 multiplies
// query rows x keys (a thread owns a row, so maximum and sum over keys stay in the thread); pass 2 multiplies
// keys x query rows - the same two shared-memory operands with their roles exchanged - so that a thread owns a
// key and the sum over the rows stays in the thread as well: it stores token scores and nothing else. (With
// rows in lanes in both passes the sum over rows was a transposing warp reduction, four instructions per element
// and four warps to meet on every panel: 15 us of a 32768-token layer's pass 2, 128 rows, against the
// special-function unit's 7; the layer went from 56.7 to 49.6 us.) Each of the four epilogue groups has an accumulator of its own, 128 keys x 128 rows.
// A KV head with more than 128 query rows is scored as two heads of 128 and the rest.
// What bounds it is the hand-over of products to the epilogue and back. With whole tiles as ring stages the issuing thread waits on
// one barrier and commits one stage per tile instead of one per 64 dims (a satisfied wait costs it 58 clocks), but the ring holds
// five tiles instead of five and a half and frees them later. Which is faster: make_token_plan.
#include "internal.h"
#include "panels.cuh"
#include "ptx.cuh"
#include "resident.cuh"

#include <math_constants.h>
#include <type_traits>

namespace chunkkv {

namespace {

constexpr int kTThreads = 576;
constexpr int kTMiscBytes = 9216;      // group records, slices, m_i, 1 / l_i
constexpr int kTPanel = 64;            // keys per epilogue panel in pass 1, query rows per step in pass 2
constexpr int kTTile = 128;            // keys per tile: both operands of a product have 128 rows
constexpr uint32_t kTHalfBytes = kTTile * 128;     // a tile's keys x 64 dims
constexpr int kTBufs = 4;              // accumulators of 128 columns: all of tensor memory, one per epilogue group

struct TokCtl {
    unsigned long long full[kRMaxStages];
    unsigned long long empty[kRMaxStages];
    unsigned long long tfull[kTBufs];
    unsigned long long tempty[kTBufs];
    unsigned long long qfull;
    int rec_count[4];                  // epilogue warps that have left their part of the CTA's record (32 rows each)
    uint32_t tmem_base;
    uint32_t tag;                      // this launch's tag (0: not known yet)
    int abort_flag;
};

struct TokArgs {
    int L, P, w, R, Hs, d;
    int n_mt;              // scoring heads per KV head (1 or 2): scoring head v scores rows [128 (v % n_mt), ...) of KV head v / n_mt
    float sl2;
    int cph, n_tiles, n_tiles_prefix, n_stages, q_box_rows, k_box_rows;
    int off_ring, off_misc;
    float* token_scores;   // [Hs][P]
    Exchange* x;           // row records as tagged words: this kernel only runs with the GPU to itself
    unsigned* exits;
    int* status;
};

// WHOLE: a ring stage is a whole tile, else 64 dims of it.
template <bool WHOLE>
__global__ void __launch_bounds__(kTThreads, 1)
token_scores_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                    const TokArgs a) {
    constexpr uint32_t IDESC = umma_idesc_bf16(128, 128);
    extern __shared__ uint8_t smem_raw[];
    __shared__ TokCtl ctl;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int KB = a.d >> 6;
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* dyn = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t q_base = smem_base;
    const uint32_t k_base = smem_base + static_cast<uint32_t>(a.off_ring);
    float* misc = reinterpret_cast<float*>(dyn + a.off_misc);
    float* rec = misc;                 // [4 groups][{max, sum}][128]
    float* slice = misc + 1024;        // [4 slices][{max, sum}][128]
    float* nrm = misc + 2048;          // [128] -m_i
    float* inv = misc + 2176;          // [128] 1 / l_i
    volatile int* abort_flag = &ctl.abort_flag;
    const uint32_t n_stages = static_cast<uint32_t>(a.n_stages);
    const uint32_t stage = WHOLE ? kTHalfBytes * static_cast<uint32_t>(KB) : kTHalfBytes;      // (64 dims after 64 dims)

    const int hs = blockIdx.x / a.cph, part = blockIdx.x - hs * a.cph;
    const int hkv = a.n_mt == 2 ? hs >> 1 : hs, row0 = a.n_mt == 2 ? (hs & 1) * 128 : 0;
    const int R = min(128, a.R - row0);              // rows of this scoring head
    const int t_begin = a.n_tiles * part / a.cph, t_end = a.n_tiles * (part + 1) / a.cph;
    const int nt = t_end - t_begin;
    const int nt2 = max(0, min(t_end, a.n_tiles_prefix) - t_begin);   // tiles of pass 2: those that hold prefix keys

    if (threadIdx.x == 0) {
        for (int s = 0; s < a.n_stages; ++s) {
            mbar_init(smem_u32(&ctl.full[s]), 1);
            mbar_init(smem_u32(&ctl.empty[s]), 1);
        }
        for (int b = 0; b < kTBufs; ++b) {
            mbar_init(smem_u32(&ctl.tfull[b]), 1);
            mbar_init(smem_u32(&ctl.tempty[b]), 4);
        }
        mbar_init(smem_u32(&ctl.qfull), 1);
        for (int i = 0; i < 4; ++i) ctl.rec_count[i] = 0;
        ctl.tag = 0u;
        ctl.abort_flag = 0;
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
    // the selection that follows is a programmatic dependent: its CTAs may be scheduled as this grid's retire;
    // this grid itself touches no global memory before its predecessor is complete
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer: the key range, twice
        if (elect_one() && nt > 0) {
            const uint32_t qbar = smem_u32(&ctl.qfull);
            mbar_arrive_expect_tx(qbar, static_cast<uint32_t>(KB * a.q_box_rows) * 128u);
            for (int kb = 0; kb < KB; ++kb)
                tma_load_3d(q_base + static_cast<uint32_t>(kb) * kRQTileBytes, &tm_q, qbar, kb * 64, row0, hkv);   // (rows past R arrive as zeros)
            const uint32_t k_bytes = static_cast<uint32_t>((WHOLE ? KB : 1) * a.k_box_rows) * 128u;
            uint32_t st = 0, st_par = 1;
            int issued = 0;
            bool ok = true;
            for (int pass = 0; pass < 2 && ok; ++pass) {
                // pass 2 walks the tiles backwards: the keys read last in pass 1 are the ones still in L2
                const int n_pass = pass == 0 ? nt : nt2;
                for (int i = 0; i < n_pass && ok; ++i) {
                    const int t = pass == 0 ? t_begin + i : t_begin + nt2 - 1 - i;
                    for (int kb = 0; kb < KB; ++kb) {
                        const uint32_t bar = smem_u32(&ctl.full[st]);
                        if (!WHOLE || kb == 0) {
                            ok = mbar_wait(smem_u32(&ctl.empty[st]), st_par, abort_flag);
                            if (!ok) break;
                            mbar_arrive_expect_tx(bar, k_bytes);
                        }
                        tma_load_3d(k_base + st * stage + (WHOLE ? kb * kTHalfBytes : 0u), &tm_k, bar, kb * 64, t * kTTile, hkv);
                        if (!WHOLE || kb == KB - 1) {
                            ++issued;
                            if (++st == n_stages) { st = 0; st_par ^= 1u; }
                        }
                    }
                }
            }
            if (!ok) {
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
            uint32_t st = 0, st_par = 0;
            for (int tg = 0; tg < nt + nt2 && ok; ++tg) {
                const int buf = tg % kTBufs, use = tg / kTBufs;
                ok = mbar_wait(smem_u32(&ctl.tempty[buf]), (use & 1) ^ 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint32_t d_addr = tmem_base + static_cast<uint32_t>(buf * 128);
                const bool keys_first = tg >= nt;        // pass 2: lanes are keys
#pragma unroll
                for (int kb = 0; kb < 2; ++kb) {
                    if (kb >= KB) break;
                    if (!WHOLE || kb == 0) {
                        ok = mbar_wait(smem_u32(&ctl.full[st]), st_par, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                    }
                    const uint64_t k_desc = umma_desc_sw128(k_base + st * stage + (WHOLE ? kb * kTHalfBytes : 0u));
                    const uint64_t q_desc = umma_desc_sw128(q_base + static_cast<uint32_t>(kb) * kRQTileBytes);
                    const uint64_t a_desc = keys_first ? k_desc : q_desc, b_desc = keys_first ? q_desc : k_desc;
#pragma unroll
                    for (int k4 = 0; k4 < 4; ++k4)
                        umma_bf16(d_addr, a_desc + 2u * k4, b_desc + 2u * k4, IDESC, (kb > 0 || k4 > 0) ? 1u : 0u);
                    if (!WHOLE) {
                        umma_commit(smem_u32(&ctl.empty[st]));
                        if (++st == n_stages) { st = 0; st_par ^= 1u; }
                    }
                }
                if (!ok) break;
                umma_commit(smem_u32(&ctl.tfull[buf]));
                if (WHOLE) {
                    umma_commit(smem_u32(&ctl.empty[st]));
                    if (++st == n_stages) { st = 0; st_par ^= 1u; }
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        const int et = threadIdx.x - 64;
        const int grp = (warp - 2) >> 2, quarter = warp & 3;
        const int row = quarter * 32 + lane;             // lane of tensor memory: query row in pass 1, key in pass 2
        const bool active = row < R;
        const int last_visible = a.P + ((row0 + row) % a.w);
        const uint32_t acc = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + static_cast<uint32_t>(grp * 128);
        int tg = grp;                                    // this group's next tile, counted over both passes; tile tg uses accumulator tg % 4
        // (behind griddepcontrol.wait; beside the first keys' way here, which the issuing thread should not wait for twice)
        if (et == 0) *const_cast<volatile uint32_t*>(&ctl.tag) = take_tag(*a.x);
        // ---- pass 1: (max, sum of exp2) per row over this CTA's keys
        float run_m = -CUDART_INF_F, run_l = 0.f;
        bool scored = true;
        for (; tg < nt; tg += kTBufs) {
            bool ready = true;
            if (lane == 0) ready = mbar_wait(smem_u32(&ctl.tfull[grp]), (tg / kTBufs) & 1, abort_flag);
            scored = __shfl_sync(0xffffffffu, ready, 0);
            if (!scored) break;
            tc_fence_after();
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                float v[kTPanel];
                load_panel<kTPanel>(acc + static_cast<uint32_t>(half * kTPanel), v);
                if (half == 1) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&ctl.tempty[grp]));
                }
                const int j0 = (t_begin + tg) * kTTile + half * kTPanel;
                float m2, l;
                auto emit = [](int, float) {};
                if (j0 + kTPanel <= a.P)
                    panel_fast<8, kTPanel>(v, a.sl2, emit, &m2, &l);
                else
                    panel_static_tail<8, kTPanel>(v, a.sl2, emit, j0, a.P, last_visible, &m2, &l);
                merge_ml(run_m, run_l, m2, l);
            }
        }
        rec[(grp * 2 + 0) * 128 + row] = active ? run_m : -CUDART_INF_F;
        rec[(grp * 2 + 1) * 128 + row] = active ? run_l : 0.f;
        // ---- the head's row statistics: the last of the warps that hold the same 32 rows merges their parts and stores them; every
        // thread then takes a quarter of the records of one row of the head, and the quarters are put together
        if (scored) {
            __threadfence_block();
            __syncwarp();
            const uint32_t tag = wait_tag(&ctl.tag, abort_flag);
            int old = 0;
            if (lane == 0) old = atomicAdd(&ctl.rec_count[quarter], 1);
            if (__shfl_sync(0xffffffffu, old, 0) == 3) {
                __threadfence_block();
                float M = -CUDART_INF_F, S = 0.f;
#pragma unroll
                for (int g = 0; g < 4; ++g) merge_ml(M, S, rec[(g * 2) * 128 + row], rec[(g * 2 + 1) * 128 + row]);
                if (tag != 0u) st_tagged2(&a.x->record[static_cast<size_t>(blockIdx.x) * 128 + row], M, S, tag);
            }
            float M = -CUDART_INF_F, S = 0.f;
            if (tag != 0u && active) {
                const ulonglong2* src = a.x->record + static_cast<size_t>(hs) * a.cph * 128 + row;
                for (int j0 = grp; j0 < a.cph; j0 += 20)             // five records in flight
                    if (!take_records<5, true>(src + j0 * 128, 4 * 128, min(5, (a.cph - j0 + 3) / 4), tag, M, S, abort_flag)) break;
            }
            slice[(grp * 2 + 0) * 128 + row] = M;
            slice[(grp * 2 + 1) * 128 + row] = S;
        }
        named_barrier(1, 512);
        const bool ok = ctl.abort_flag == 0;         // same answer in every epilogue thread
        if (ok) {
            if (et < 128) {
                float M2 = -CUDART_INF_F, L2 = 0.f;
#pragma unroll
                for (int q = 0; q < 4; ++q) merge_ml(M2, L2, slice[(q * 2) * 128 + et], slice[(q * 2 + 1) * 128 + et]);
                nrm[et] = -M2;
                inv[et] = et < R ? 1.0f / L2 : 0.f;
            }
            named_barrier(1, 512);
            // ---- pass 2: the same tiles again, backwards, keys in lanes: normalised and summed over the rows
            float* out = a.token_scores + static_cast<size_t>(hs) * a.P;
            const unsigned long long s2 = pack2(a.sl2, a.sl2);
            const int n_half = R > kTPanel ? 2 : 1;
            // A key's sum over the rows r0 .. r0 + 63 of this scoring head, as eight chains of eight terms added as a tree. A
            // column past R is left out by selection, not by a factor 0: it is the product of a zero row, which is NaN for a
            // key with an infinite component.
            auto sum_rows = [&](auto all, int r0, const float (&v)[kTPanel]) -> float {
                constexpr bool ALL = decltype(all)::value;               // every one of the 64 rows exists
                const float4* n4 = reinterpret_cast<const float4*>(nrm + r0);
                const float4* i4 = reinterpret_cast<const float4*>(inv + r0);
                unsigned long long sum[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
                for (int u = 0; u < kTPanel / 4; ++u) {
                    const int left = ALL ? 4 : R - r0 - 4 * u;           // rows of this group of four
                    if (left <= 0) break;
                    const float4 n = n4[u], iv = i4[u];                  // (the same address in every lane)
                    float x0, x1, x2, x3;
                    unpack2(fma2(pack2(v[4 * u], v[4 * u + 1]), s2, pack2(n.x, n.y)), x0, x1);
                    unpack2(fma2(pack2(v[4 * u + 2], v[4 * u + 3]), s2, pack2(n.z, n.w)), x2, x3);
                    const float e0 = ex2_approx(x0), e1 = left > 1 ? ex2_approx(x1) : 0.f;
                    const float e2 = left > 2 ? ex2_approx(x2) : 0.f, e3 = left > 3 ? ex2_approx(x3) : 0.f;
                    unsigned long long* a2 = &sum[2 * (u & 1)];
                    a2[0] = fma2(pack2(e0, e1), pack2(iv.x, iv.y), a2[0]);
                    a2[1] = fma2(pack2(e2, e3), pack2(iv.z, iv.w), a2[1]);
                }
                float lo, hi;
                unpack2(add2(add2(sum[0], sum[1]), add2(sum[2], sum[3])), lo, hi);
                return lo + hi;
            };
            for (; tg < nt + nt2; tg += kTBufs) {
                bool ready = true;
                if (lane == 0) ready = mbar_wait(smem_u32(&ctl.tfull[grp]), (tg / kTBufs) & 1, abort_flag);
                if (!__shfl_sync(0xffffffffu, ready, 0)) break;
                tc_fence_after();
                float t = 0.f;
                for (int half = 0; half < n_half; ++half) {
                    float v[kTPanel];
                    load_panel<kTPanel>(acc + static_cast<uint32_t>(half * kTPanel), v);
                    if (half == n_half - 1) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&ctl.tempty[grp]));
                    }
                    t += (half + 1) * kTPanel <= R ? sum_rows(std::true_type{}, half * kTPanel, v) : sum_rows(std::false_type{}, half * kTPanel, v);
                }
                const int j = (t_begin + nt2 - 1 - (tg - nt)) * kTTile + row;
                if (j < a.P) out[j] = t;
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    if (threadIdx.x == 0) {
        if (ctl.abort_flag) atomicExch(a.status, 1);
        if (ctl.tag == kLastTag && atomicAdd(a.exits, 1u) + 1u == gridDim.x) {
            *a.exits = 0u;
            end_tags(*a.x);
            __threadfence();
        }
    }
}

}  // namespace

bool make_token_plan(int L, int w, int R, int Hkv, int d, int max_ctas, int smem_limit, TokenPlan* plan) {
    const int n_mt = R > 128 ? 2 : 1, Hs = Hkv * n_mt;
    if (R < 1 || R > 256 || (d != 64 && d != 128) || L < 1 || L - w < 1 || Hs < 1 || Hs > kResidentMaxHeads) return false;
    if (max_ctas < Hs) return false;
    TokenPlan p{};
    p.n_mt = n_mt;
    p.Hs = Hs;
    p.cph = (max_ctas < kExchangeCtas ? max_ctas : kExchangeCtas) / Hs;
    p.grid = p.cph * Hs;
    p.n_tiles = (L + kTTile - 1) / kTTile;
    p.n_tiles_prefix = (L - w + kTTile - 1) / kTTile;
    const int KB = d / 64;
    const int q_bytes = KB * kRQTileBytes;
    const int fixed = 1024 + q_bytes + 1024 + kTMiscBytes;
    // Whole tiles as stages for one scoring head a KV head and more than ten tiles a CTA, us with stages of 64 dims -> of whole
    // tiles, d = 128, with the chunk sums: 8 heads, 128 rows 32768 tokens 40.3 -> 39.6, 46657 51.1 -> 50.0, 90000 79 -> 76.4; 4 heads, 112 rows
    // 56490 37.3 -> 36.5. Not for less: 8 heads, 64 rows 16000 22.8 -> 23.1; 4 heads, 112 rows 32768 29.1 -> 29.5, 46657 (ten tiles) 34.9 -> 35.2;
    // nor for the two scoring heads of more than 128 rows: 4 heads, 224 rows 46657 41.1 -> 41.5, 8 heads, 256 rows 32768 51.5 -> 52.0.
    p.whole = KB == 1 || (n_mt == 1 && p.n_tiles > 10 * p.cph);
    const int stage = (p.whole ? KB : 1) * static_cast<int>(kTHalfBytes);
    int ns = (smem_limit - fixed) / stage;
    if (ns > kRMaxStages) ns = kRMaxStages;
    if (ns < (p.whole ? 2 : 2 * KB)) return false;
    p.n_stages = ns;
    p.off_ring = q_bytes;
    p.off_misc = p.off_ring + ns * stage + 1024;
    p.smem_bytes = 1024 + p.off_misc + kTMiscBytes;
    *plan = p;
    return true;
}

cudaError_t launch_token_scores(const TokenPlan& plan, const CUtensorMap& tm_q, const CUtensorMap& tm_k,
                                const TokenIO& io, cudaStream_t stream) {
    TokArgs a{};
    a.L = io.L; a.P = io.L - io.w; a.w = io.w; a.R = io.R; a.Hs = plan.Hs; a.d = io.d; a.n_mt = plan.n_mt;
    a.sl2 = io.sl2;
    a.cph = plan.cph; a.n_tiles = plan.n_tiles; a.n_tiles_prefix = plan.n_tiles_prefix; a.n_stages = plan.n_stages;
    a.q_box_rows = 128;                  // (rows past R arrive as zeros)
    a.k_box_rows = io.L < kTTile ? io.L : kTTile;
    a.off_ring = plan.off_ring; a.off_misc = plan.off_misc;
    a.token_scores = io.token_scores;
    a.x = io.exchange;
    a.exits = io.counters;
    a.status = io.status;
    const void* kern = plan.whole ? reinterpret_cast<const void*>(token_scores_kernel<true>) : reinterpret_cast<const void*>(token_scores_kernel<false>);
    static int smem_all[2][64] = {{0}};
    int* smem_set = smem_all[plan.whole ? 1 : 0];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || smem_set[dev] < plan.smem_bytes) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, plan.smem_bytes);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) smem_set[dev] = plan.smem_bytes;
    }
    void* params[] = {const_cast<CUtensorMap*>(&tm_q), const_cast<CUtensorMap*>(&tm_k), &a};
    // The CTAs of a head wait for one another, so all must be resident: the plan allows at most one CTA
    // per SM (its shared memory) and no more CTAs than SMs, and this path is only taken with the whole
    // GPU, so every CTA becomes resident without waiting for another CTA of this grid. Launched as a
    // programmatic dependent of the preceding kernel, the set-up of this one overlaps the end of that one.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(plan.grid);
    cfg.blockDim = dim3(kTThreads);
    cfg.dynamicSmemBytes = static_cast<size_t>(plan.smem_bytes);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, kern, params);
}

}  // namespace chunkkv
