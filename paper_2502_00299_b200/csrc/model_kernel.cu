// Many layers in one launch (ChunkKV Algorithm 2: "for l = 0 .. N_layers - 1", with Algorithm 3 per
// computed layer): a persistent version of the layer kernel of layer_resident.cu in which the
// steps of successive layers overlap inside every CTA.
//
// A CTA belongs to one KV head and one key range for the whole launch. A KV head with more than 128
// query rows has two query tiles: each key tile is loaded once and multiplied with both. The CTA's
// (key tile, query tile) products are "virtual tiles" in issue order; its panels (half a virtual
// tile each) are numbered through the launch, and a panel's accumulator, epilogue group and ring slot
// all follow from that number. Its warps have roles:
//   warp 0         TMA producer: streams the Q tile and the CTA's K tiles of layer after layer
//                  through the shared-memory ring, as far ahead as the ring allows
//   warp 1         tcgen05.mma issuer
//   warps 2..17    epilogue, four groups of four warps: one exponential per score element, chunk sums
//                  into a ring of tensor-memory columns that holds more than one layer (the part of
//                  the ring that does not fit there lies in scratch: long contexts, small chunks); at the end
//                  of a layer a group leaves its per-row (max, sum) in shared memory and goes straight
//                  on with the next layer; when the head's row statistics have arrived (normally long
//                  before they are needed) it contracts the partial sums it wrote itself over the rows
//                  into chunk scores of the CTA's key range (global memory)
//   warp 18        for each computed layer, once a selector CTA has published the head's
//                  kept-chunk list, moves this CTA's share of the kept K/V rows with bulk asynchronous
//                  copies (global -> shared -> global, whole chunks at a time) - for the computed
//                  layer and for every following layer that reuses its indices
//   warp 19        announces the CTA's record of row statistics, which the last of the epilogue warps that hold the same
//                  32 rows stores, waits (bounded) for the head's other CTAs - the epilogue threads merge the head's
//                  records for the contraction - and announces the CTA's chunk scores when they are stored
// The CTAs after the scoring CTAs are selectors: exact top-k per head, out_idx, kept-chunk lists.
//
// So while the selectors and copy threads work on layer l, the other warps already score layer l + 1:
// the latency-bound steps cost no memory bandwidth and the copies ride along with the K stream.
// Hand-over counters only grow during a launch (layer l waits for (l + 1) x CTAs arrivals); the
// last CTA to leave clears them. Every wait is bounded and reports through the device status word.
#include "internal.h"
#include "panels.cuh"
#include "ptx.cuh"
#include "resident.cuh"
#include "select.cuh"

#include <math_constants.h>

namespace chunkkv {

namespace {

constexpr int kMThreads = 640;          // warp 0: TMA, warp 1: UMMA issue, warps 2..17: epilogue, warp 18: row copies, warp 19: row statistics
                                        // (five warps per scheduler: a sixth would cut every thread to 80 registers)
constexpr int kMMiscBytes = 16384;      // epilogue: group records (two slots), m_i, 1 / l_i, row sums per lane quarter
constexpr int kMSlots = 8;              // most staging slots of the row copies
constexpr int kMBlkSlots = 32;          // room for the chunk slots of one contraction block
// Tensor memory, small variant: three 64-column accumulators (one 60-key panel of a tile each, in rotation; the
// second panel of a tile is computed on keys 56 .. 119 so that its operand starts on a swizzle-atom
// boundary, and begins at column 4), and 320 columns of chunk partial sums: a ring that holds one
// layer and two thirds of the next at c = 10, so the statistics of a layer have most of the next
// layer's scoring time to travel before its contraction needs them.
// Big variant: two 128-column accumulators (a whole virtual tile each, one per pair of epilogue groups) and 256
// columns of the ring, which continues in scratch. Half as many products to issue, each at the tensor pipe's rate
// (an N = 64 product takes 48 clocks, an N = 128 one 64: the query tile is read from shared memory for each), which
// two query tiles need: with three 64-column accumulators a 256-row layer spent 45 % of its time waiting for products.
constexpr int kMAccN = 64;
constexpr int kMAccBufs = 3;
constexpr int kMAccSlots = 12;                     // (buffer, epilogue group) pairs: lcm(3 buffers, 4 groups)
constexpr int kMAcc1Row = 56;
__host__ __device__ constexpr int model_part_col0(bool big) { return big ? 2 * kRUmmaN : kMAccBufs * kMAccN; }
// Ring sizes are multiples of the four epilogue groups: a panel's ring slot is its number (since the
// start of the launch) modulo the ring size and its group is that number modulo 4, so a ring slot
// is only ever reused by the group that wrote and contracted its previous contents. Panels held on chip:
// the small variant keeps panel maxima in shared memory (a row set per panel: at most 84 panels, fewer where
// more would only cost ring stages), the big one beside the sums in tensor memory.
__host__ __device__ constexpr int model_ring_panels(int c, bool big) {
    const int spp = panel_keys(c) / c;
    const int fit = (512 - model_part_col0(big)) / (big ? spp + 1 : spp) / 4 * 4;
    return big ? fit : (c >= 32 ? 64 : (c == 16 ? 72 : (fit > 84 ? 84 : fit)));
}
// Staging slots of the row copies: as many as fit about 40 KB (a slot holds a chunk's K and V rows)
__host__ __device__ constexpr int model_copy_slots(int c, int d) {
    const int n = 40960 / (4 * c * d);
    return n > kMSlots ? kMSlots : (n < 3 ? 3 : n);
}
constexpr int kBarGroup = 2;                       // named barriers 2 .. 5: the four warps of an epilogue group

struct ModelCtl {
    unsigned long long full[kRMaxStages];
    unsigned long long empty[kRMaxStages];
    unsigned long long tfull[kMAccSlots];      // by panel number modulo 12: one (accumulator, epilogue group) pair each
                                               // (big variant: the first two, one per accumulator)
    unsigned long long tempty[kMAccSlots];
    unsigned long long qfull;
    unsigned long long qempty;
    unsigned long long gfull[kMSlots];
    unsigned long long sfull;          // a kept-chunk list has landed in shared memory (copy thread)
    unsigned long long stat_full[2];   // m_i and 1 / l_i of a slot are in shared memory (statistics warps -> epilogue)
    unsigned long long pub_done[2];    // the slot's record is stored, 32 rows an arrival (-> statistics warp)
    unsigned long long sc_done[2];     // every epilogue warp has stored its chunk scores of the slot (-> statistics warp)
    int pub_count[2][2][4];            // epilogue warps that have left their part of a slot's record: [slot parity][query tile][32 rows]
    uint32_t tmem_base;
    int abort_flag;
    int sel_flag[2];                   // selector CTAs: wait result, abort flag
};

struct ModelLayer {
    const uint4* K;
    const uint4* V;
    uint4* out_K;
    uint4* out_V;
    int32_t* out_idx;
    int slot;          // computed layer: its slot (0 .. n_compute - 1); reuse layer: the slot of its source layer
    int computes;      // 1: scored and selected here; 0: gathered with the slot's indices
};

struct ModelParams {
    CUtensorMap tm_q[kModelMaxCompute];
    CUtensorMap tm_k[kModelMaxCompute];
    ModelLayer layer[kModelMaxLayers];
    int n_layers, n_compute;
    int L, P, w, R, d;
    int n_mt;              // 128-row query tiles per KV head (1 or 2)
    float sl2;
    int cph, n_tiles, n_stages, q_box_rows, k_box_rows;
    int C, k, n_max, Hkv;
    int Cpad;              // row stride of the chunk scores (C rounded up to a multiple of 4: rows stay 16-byte aligned)
    int n_score, n_sel;    // scoring CTAs (Hkv * cph) and selector CTAs (the rest of the grid)
    int strided;           // rows of a head are not adjacent in memory: kept rows are fetched through tm_rk / tm_rv
    int copy_box_bytes;    // bytes of such a box
    int ring_on, ring;     // big variant: panels of the ring in tensor memory, panels of the ring in all
    int spill_rows;        // rows of a panel's record in scratch (whole warps)
    int ahead, stride;     // big variant: own panels of a layer that a group scores before the contraction of the layer before,
                           // and between two blocks of it
    int copy_slots;
    int sel_row_bytes;     // bytes of one kept-chunk list: 4 header ints + the kept chunk ids, padded to 16 bytes
    int sel_keys_fit;      // selector: the keys of a head fit its shared memory (many chunks per thread)
    int off_ring, off_pmax, off_misc, off_tail, stage_slot_bytes;
    float* cta_stat;       // [2 (slot parity)][grid][n_mt][{max, sum}][128]
    float* scores;         // [n_compute][Hkv][n_mt][Cpad]
    float* spill;          // per scoring CTA: [ring - ring_on][rows / 32][chunk sums, panel maximum][32 rows], and the blocks of warps without rows
    unsigned* cnt_a;       // [Hkv]
    unsigned* cnt_b;       // [Hkv]  chunk scores of a slot announced by the scoring CTAs
    unsigned* cnt_c;       // [Hkv]  kept-chunk lists announced by the selector CTAs
    int* sel_rows;         // [n_compute][Hkv][sel_row_bytes / 4]
    unsigned* exits;
    int* status;
    // strided caches: boxes of one chunk's rows of K and of V, per layer (a launch takes at most kModelMaxStrided then)
    CUtensorMap tm_rk[kModelMaxStrided];
    CUtensorMap tm_rv[kModelMaxStrided];
};
static_assert(sizeof(ModelParams) <= 32764, "kernel parameters");

// ---- bulk asynchronous copies (no multicast): global -> this CTA's shared memory with byte-counted
//      completion on an mbarrier, and shared -> global in bulk groups
__device__ __forceinline__ void bulk_load(uint32_t dst_smem, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst_smem),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, uint32_t src_smem, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src_smem), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Bounded wait of a whole warp on a counter that only grows: every lane performs the acquire load, so
// each lane's later loads are ordered behind the arrivals it has seen. Lane 0 keeps the time limit.
__device__ __forceinline__ bool wait_counter_warp(const unsigned* counter, unsigned target, volatile int* abort_flag) {
    const long long t0 = clock64();
    for (;;) {
        unsigned cur;
        asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(cur) : "l"(counter) : "memory");
        if (__all_sync(0xffffffffu, cur >= target)) return true;
        int bad = 0;
        if ((threadIdx.x & 31) == 0) {
            if (*abort_flag) bad = 1;
            else if (clock64() - t0 > kWaitLimitClocks) { *abort_flag = 1; bad = 1; }
        }
        if (__shfl_sync(0xffffffffu, bad, 0)) return false;
    }
}

// Bounded wait of one thread on a counter that only grows.
__device__ __forceinline__ bool wait_counter(const unsigned* counter, unsigned target, volatile int* abort_flag,
                                             unsigned sleep_ns) {
    unsigned cur;
    asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(cur) : "l"(counter) : "memory");
    if (cur >= target) return true;
    const long long t0 = clock64();
    for (;;) {
        if (sleep_ns) __nanosleep(sleep_ns);
        asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(cur) : "l"(counter) : "memory");
        if (cur >= target) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > kWaitLimitClocks) { *abort_flag = 1; return false; }
    }
}

// Selector CTA (the CTAs after the scoring CTAs; they run on SMs the scoring grid leaves free): for
// every slot and each of its KV heads, once the head's chunk scores are complete, the whole CTA
// runs the exact top-k (select.cuh), writes the kept positions to out_idx of the computed layer
// and of every layer that reuses its indices (and zero rows behind the kept rows, which exist
// only when the clipped last chunk is kept), publishes the kept-chunk list for the scoring CTAs'
// copy threads and announces it on the head's third counter.
template <int C_STATIC, SelectIn WHERE>
__device__ __forceinline__ bool selector_loop(const ModelParams& p, uint8_t* dyn, int* flag_smem) {
    SelectSmem& ss = *reinterpret_cast<SelectSmem*>(dyn);
    constexpr size_t kSelBytes = (sizeof(SelectSmem) + 127) & ~size_t(127);
    uint32_t* kbuf = reinterpret_cast<uint32_t*>(dyn + kSelBytes);    // keys, when there are many chunks per thread
    const int sid = static_cast<int>(blockIdx.x) - p.n_score;
    const int kk = min(p.k, p.C);
    const int row_ints = p.sel_row_bytes / 4;
    volatile int* flag = flag_smem;
    for (int li = 0; li < p.n_layers;) {
        const int s = p.layer[li].slot;
        int lj_end = li + 1;
        while (lj_end < p.n_layers && !p.layer[lj_end].computes) ++lj_end;
        for (int hkv = sid; hkv < p.Hkv; hkv += p.n_sel) {
            if (threadIdx.x == 0) {
                const unsigned target = static_cast<unsigned>(s + 1) * p.cph;
                flag[0] = wait_counter(p.cnt_b + hkv, target, flag + 1, 100) ? 1 : 0;      // (acquires; the barrier passes it on)
            }
            __syncthreads();
            if (!flag[0]) return false;
            const float* sc = p.scores + (static_cast<size_t>(s) * p.Hkv + hkv) * p.n_mt * p.Cpad;
            const float* sc2 = p.n_mt == 2 ? sc + p.Cpad : nullptr;
            if (p.sel_keys_fit || p.C <= kMThreads * select_reg_keys(WHERE))
                select_kept<WHERE>(sc, sc2, p.C, p.k, ss, kbuf);
            else
                select_head_rows(sc, sc2, p.L, p.w, C_STATIC, p.C, p.k, p.n_max, p.layer[li].out_idx + static_cast<size_t>(hkv) * p.n_max,
                                 ss, nullptr);
            const int n_tok = select_tokens(p.P, C_STATIC, p.C, p.k, ss);
            // the kept-chunk list for the copy warps: [n_tok, -, -, -, chunk ids]. It is announced before the positions are written, which nothing
            // in this launch reads, and by another warp than the one that waits for the next head: a release waits for the stores before it.
            int* row = p.sel_rows + (static_cast<size_t>(s) * p.Hkv + hkv) * row_ints;
            if (threadIdx.x == 0) row[0] = n_tok;
            for (int r = threadIdx.x; r < kk; r += kMThreads) row[4 + r] = ss.sel[r];
            __syncthreads();
            if (threadIdx.x == kMThreads - 32)      // release: the list is visible to whoever sees the count
                asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p.cnt_c + hkv) : "memory");
            const int vpr = p.d >> 3;
            for (int n = threadIdx.x; n < p.n_max; n += kMThreads) {
                const int pos = select_position(ss, n, n_tok, C_STATIC, p.P, p.w);
                for (int lj = li; lj < lj_end; ++lj) p.layer[lj].out_idx[static_cast<size_t>(hkv) * p.n_max + n] = pos;
            }
            const int nz = (p.n_max - n_tok - p.w) * vpr;
            if (nz > 0)
                for (int lj = li; lj < lj_end; ++lj) {
                    uint4* zk = p.layer[lj].out_K + (static_cast<size_t>(hkv) * p.n_max + n_tok + p.w) * vpr;
                    uint4* zv = p.layer[lj].out_V + (static_cast<size_t>(hkv) * p.n_max + n_tok + p.w) * vpr;
                    for (int i = threadIdx.x; i < nz; i += kMThreads) { zk[i] = make_uint4(0, 0, 0, 0); zv[i] = make_uint4(0, 0, 0, 0); }
                }
        }
        li = lj_end;
    }
    return true;
}

// BIG: two query tiles, or a ring that reaches into scratch. A variant of its own, so that the kernel for up to 128 rows
// carries none of it.
template <int C_STATIC, bool BIG>
__global__ void __launch_bounds__(kMThreads, 1)
model_kernel(const __grid_constant__ ModelParams p) {
    constexpr int WP = panel_keys(C_STATIC);
    constexpr int TILE = 2 * WP;
    constexpr uint32_t STAGE = TILE * 128;
    constexpr int SPP = WP / C_STATIC;
    constexpr int ACC1 = WP == 64 ? 64 : kMAcc1Row;       // first key of a tile's second product (a swizzle-atom boundary)
    constexpr int COL1 = WP - ACC1;                       // accumulator column its panel begins at
    constexpr int PART0 = model_part_col0(BIG);
    constexpr uint32_t IDESC = umma_idesc_bf16(128, BIG ? kRUmmaN : kMAccN);

    extern __shared__ uint8_t smem_raw[];
    __shared__ ModelCtl ctl;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int KB = p.d >> 6;
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* dyn = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t q_base = smem_base;
    const uint32_t k_base = smem_base + static_cast<uint32_t>(p.off_ring);
    float* pmax = reinterpret_cast<float*>(dyn + p.off_pmax);
    float* misc = reinterpret_cast<float*>(dyn + p.off_misc);
    float* rec = misc;                 // [4 groups][{max, sum}][128]; the odd slots' copy sits at misc + 3072
    float* gstat = misc + 1024;        // [4 groups][{m_i, 1 / l_i}][128]
    float* red = misc + 2048;          // [4 groups][block parity][4 lane quarters][kMBlkSlots]
    volatile int* abort_flag = &ctl.abort_flag;
    const uint32_t n_stages = static_cast<uint32_t>(p.n_stages);

    if (static_cast<int>(blockIdx.x) >= p.n_score) {
        // ------------------------------------------------------------------ selector CTA
        if (threadIdx.x == 0) { ctl.sel_flag[0] = 1; ctl.sel_flag[1] = 0; }
        __syncthreads();
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const bool s_ok = selector_loop<C_STATIC, BIG && C_STATIC == 8 ? kSelModelCore : kSelModel>(p, dyn, ctl.sel_flag);
        __syncthreads();
        if (threadIdx.x == 0) {
            if (!s_ok) atomicExch(p.status, 1);
            const unsigned old = atomicAdd(p.exits, 1u);
            if (old + 1u == gridDim.x) {
                for (int h = 0; h < p.Hkv; ++h) { p.cnt_a[h] = 0u; p.cnt_b[h] = 0u; p.cnt_c[h] = 0u; }
                *p.exits = 0u;
                __threadfence();
            }
        }
        return;
    }
    const int hkv = blockIdx.x / p.cph, part = blockIdx.x - hkv * p.cph;
    // tiles are dealt out rounding up, so the head's last CTA - whose last panels take the slow, masked path -
    // is never one of those that get an extra tile
    const int t_begin = (p.n_tiles * part + p.cph - 1) / p.cph, t_end = (p.n_tiles * (part + 1) + p.cph - 1) / p.cph;
    const int nt = t_end - t_begin;
    const int n_mt = BIG ? p.n_mt : 1;
    const bool two = n_mt == 2;
    const int n_vt = two ? 2 * nt : nt;              // virtual tiles of this CTA per layer

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.n_stages; ++s) {
            mbar_init(smem_u32(&ctl.full[s]), 1);
            mbar_init(smem_u32(&ctl.empty[s]), 1);
        }
        for (int b = 0; b < kMAccSlots; ++b) {
            mbar_init(smem_u32(&ctl.tfull[b]), 1);
            mbar_init(smem_u32(&ctl.tempty[b]), BIG ? 8 : 4);      // one arrival per reading warp
        }
        mbar_init(smem_u32(&ctl.qfull), 1);
        mbar_init(smem_u32(&ctl.qempty), 1);
        for (int s = 0; s < kMSlots; ++s) mbar_init(smem_u32(&ctl.gfull[s]), 1);
        mbar_init(smem_u32(&ctl.sfull), 1);
        mbar_init(smem_u32(&ctl.stat_full[0]), 1);
        mbar_init(smem_u32(&ctl.stat_full[1]), 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&ctl.pub_done[b]), 4 * n_mt);
            mbar_init(smem_u32(&ctl.sc_done[b]), 16);
        }
        for (int i = 0; i < 16; ++i) (&ctl.pub_count[0][0][0])[i] = 0;
        ctl.abort_flag = 0;
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
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (elect_one() && nt > 0) {
            const uint32_t qbar = smem_u32(&ctl.qfull);
            const uint32_t q_bytes = static_cast<uint32_t>(n_mt * KB * p.q_box_rows) * 128u;
            const uint32_t k_bytes = static_cast<uint32_t>(p.k_box_rows) * 128u;
            // The keys, which are read once, leave the L2 first where the ring continues in scratch (30000 tokens, 128 rows, c = 5 222 -> 217 us,
            // 256 rows, c = 10 246 -> 241) and where a layer has few of them (224 rows, 4 heads: 2300 tokens, c = 16 266.6 -> 258.7, 5500 tokens, c = 20
            // 169.4 -> 166.5). Not otherwise: the row copies of the next layer read the kept key rows again (16000 tokens, 16 MB, c = 20,
            // 10 % kept: 315.4 -> 317.1).
            const bool leave = p.ring > p.ring_on || 2ll * p.Hkv * p.L * p.d <= (6ll << 20);
            const uint64_t policy = leave ? l2_policy_evict_first() : l2_policy_evict_normal();
            uint32_t st = 0, st_par = 1;
            int issued = 0;
            bool ok = true;
            // A layer's first key tiles go ahead of its queries: the Q tile is free only when the last product of the layer before has
            // read it, and by then the stages that were free earlier hold keys. Before this, the K stream stopped at every layer until the
            // ring had run empty (5.5k of 30.5k clocks a layer of 32768 tokens, 128 rows). As many stages as are not the layer before's last tile
            // (its products end together with the Q tile's use).
            const int n_k = nt * KB, q_at = min(n_k, p.n_stages - KB);
            for (int s = 0; s < p.n_compute && ok; ++s) {
                prefetch_tmap(&p.tm_q[s]);
                prefetch_tmap(&p.tm_k[s]);
                for (int mt = 0; mt < n_mt; ++mt)
                    for (int kb = 0; kb < KB; ++kb) tma_prefetch_3d(&p.tm_q[s], kb * 64, mt * 128, hkv);
                int t = t_begin, kb = 0;
                for (int i = 0; i <= n_k; ++i) {
                    if (i == (s == 0 ? 0 : q_at)) {
                        if (s > 0) ok = mbar_wait(smem_u32(&ctl.qempty), (s - 1) & 1, abort_flag);
                        if (!ok) break;
                        mbar_arrive_expect_tx(qbar, q_bytes);
                        for (int mt = 0; mt < n_mt; ++mt)    // (rows past R of the second tile arrive as zeros)
                            for (int b = 0; b < KB; ++b)
                                tma_load_3d(q_base + static_cast<uint32_t>(mt * KB + b) * kRQTileBytes, &p.tm_q[s], qbar, b * 64, mt * 128, hkv);
                    }
                    if (i == n_k) break;
                    ok = mbar_wait(smem_u32(&ctl.empty[st]), st_par, abort_flag);
                    if (!ok) break;
                    const uint32_t bar = smem_u32(&ctl.full[st]);
                    mbar_arrive_expect_tx(bar, k_bytes);
                    if constexpr (BIG) tma_load_3d_hint(k_base + st * STAGE, &p.tm_k[s], bar, kb * 64, t * TILE, hkv, policy);
                    else tma_load_3d(k_base + st * STAGE, &p.tm_k[s], bar, kb * 64, t * TILE, hkv);
                    ++issued;
                    if (++st == n_stages) { st = 0; st_par ^= 1u; }
                    if (++kb == KB) { kb = 0; ++t; }
                }
            }
            if (!ok) {
                const int back = min(issued, p.n_stages);
                for (int i = 1; i <= back; ++i) {
                    const int cc = issued - i, s = cc % p.n_stages;
                    const long long t0 = clock64();
                    while (!mbar_try_wait(smem_u32(&ctl.full[s]), (cc / p.n_stages) & 1) &&
                           clock64() - t0 < kWaitLimitClocks / 8) {
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ UMMA issuer
        if (elect_one() && nt > 0) {
            const uint64_t q_desc = umma_desc_sw128(q_base), k_desc = umma_desc_sw128(k_base);
            const bool both = KB == 2;                   // d is 64 or 128: one or two stages a tile
            uint32_t st = 0, st_par = 0;
            uint32_t buf = 0, aslot = 0, e_slot = kMAccSlots - kMAccBufs, e_par = 1;   // small: accumulator, (accumulator, group) slot; slot to wait for
            int vg = 0;                  // virtual tiles issued so far (all layers); the epilogue pair vg & 1 reads tile vg
            bool ok = true;
            for (int s = 0; s < p.n_compute && ok; ++s) {
                ok = mbar_wait(smem_u32(&ctl.qfull), s & 1, abort_flag);
                for (int ti = 0; ti < nt && ok; ++ti) {
                    const uint32_t s0 = st, p0 = st_par;
                    if (++st == n_stages) { st = 0; st_par ^= 1u; }
                    const uint32_t s1 = both ? st : s0, p1 = both ? st_par : p0;
                    if (both && ++st == n_stages) { st = 0; st_par ^= 1u; }
                    const uint32_t full0 = smem_u32(&ctl.full[s0]), full1 = smem_u32(&ctl.full[s1]);
                    if constexpr (BIG) {
                        for (int mt = 0; mt < n_mt; ++mt, ++vg) {
                            const uint32_t ab = vg & 1;
                            const uint32_t tempty = smem_u32(&ctl.tempty[ab]), te_par = ((vg >> 1) & 1) ^ 1;
                            ok = mt == 0 ? mbar_wait3(full0, p0, full1, p1, tempty, te_par, abort_flag) : mbar_wait(tempty, te_par, abort_flag);
                            if (!ok) break;
                            tc_fence_after();
                            issue_products(tmem_base + ab * kRUmmaN, q_desc + static_cast<uint32_t>(mt * KB) * (kRQTileBytes >> 4),
                                           k_desc + s0 * (STAGE >> 4), k_desc + s1 * (STAGE >> 4), both, IDESC);
                            umma_commit(smem_u32(&ctl.tfull[ab]));
                        }
                    } else {
#pragma unroll
                        for (int half = 0; half < 2; ++half) {
                            // a panel goes to accumulator (panel number % 3), which the third panel before it used last:
                            // wait until that one's group has read it (the first three panels find a fresh barrier)
                            const uint32_t tempty = smem_u32(&ctl.tempty[e_slot]);
                            ok = half == 0 ? mbar_wait3(full0, p0, full1, p1, tempty, e_par, abort_flag) : mbar_wait(tempty, e_par, abort_flag);
                            if (++e_slot == kMAccSlots) { e_slot = 0; e_par ^= 1u; }
                            if (!ok) break;
                            tc_fence_after();
                            const uint32_t half_off = static_cast<uint32_t>(half * ACC1 * 128) >> 4;
                            issue_products(tmem_base + buf * kMAccN, q_desc, k_desc + s0 * (STAGE >> 4) + half_off, k_desc + s1 * (STAGE >> 4) + half_off,
                                           both, IDESC);
                            umma_commit(smem_u32(&ctl.tfull[aslot]));
                            if (++buf == kMAccBufs) buf = 0;
                            if (++aslot == kMAccSlots) aslot = 0;
                        }
                    }
                    if (!ok) break;
                    umma_commit(smem_u32(&ctl.empty[s0]));
                    if (both) umma_commit(smem_u32(&ctl.empty[s1]));
                }
                if (ok) umma_commit(smem_u32(&ctl.qempty));       // every UMMA of this layer has read the Q tile
            }
        }
    } else if (warp < 18) {
        // ------------------------------------------------------------------ epilogue
        // The chunk partial sums and panel maxima of a layer live in rings (tensor-memory columns,
        // shared memory, scratch) that hold more than one layer's worth, so after its last tile of layer s a
        // thread only publishes the CTA's row records and goes straight on with layer s + 1; the chunk scores
        // of layer s are formed between its panels.
        const int grp = (warp - 2) >> 2, quarter = warp & 3;
        const int gt = threadIdx.x - 64 - grp * 128;    // 0 .. 127 within the group
        const int pair = grp >> 1, half = grp & 1;
        const int row = quarter * 32 + lane;             // row of the query tile = lane of tensor memory
        const int qrow = row + (two ? pair * 128 : 0);   // row of the KV head (two query tiles: a pair takes one of them)
        const bool active = qrow < p.R;
        const int last_visible = p.P + (qrow % p.w);
        const uint32_t lane_addr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        const int n_pl = 2 * n_vt;
        const int PR = BIG ? p.ring : model_ring_panels(C_STATIC, false);          // panels in the ring
        constexpr int PCOLS = BIG ? SPP + 1 : SPP;                                  // tensor-memory columns of a panel
        const int ch0 = t_begin * (TILE / C_STATIC);
        const uint64_t keep = l2_policy_evict_last(), drop = l2_policy_evict_first();
        // A panel's record in scratch: a block of 32 rows for every warp that has rows, with constant offsets inside it. A warp
        // that has none does the same with one block of its own behind the records (it would cost the others more to branch).
        float* spill = nullptr;
        int spill_step = 0;                              // between the records of two ring slots
        if constexpr (BIG) {
            const int off = p.ring - p.ring_on, n_w = p.spill_rows / 32;
            const size_t cta = static_cast<size_t>(blockIdx.x) * (static_cast<size_t>(off) * n_w + 4 * (4 - n_w)) * (PCOLS * 32);
            const bool have_rows = quarter < n_w;
            spill = p.spill + cta + (have_rows ? quarter : off * n_w + grp * (4 - n_w) + quarter - n_w) * (PCOLS * 32);
            spill_step = have_rows ? PCOLS * p.spill_rows : 0;
        }
        bool ok = true;
        float run_m = -CUDART_INF_F, run_l = 0.f;
        // Contraction of a layer's partial sums into chunk scores, one block of panels at a time, between the panels of the next
        // layer: a group contracts the panels it scored itself - every thread reads back the tensor-memory columns (or
        // scratch) it wrote - so the only synchronisation is among the group's four warps (the four lane quarters of a
        // sum). It starts once `ahead` of the group's own panels of the next layer are scored, so that the row statistics
        // have arrived, and goes on block by panel, so that the groups' round trips and shuffles overlap the other groups'
        // exponentials. A block holds more panels than are scored between two blocks, and the ring more than a layer and
        // `ahead` panels per group: a slot is contracted before it is written again. (Big variant: `stride` panels between
        // two blocks and the groups a part of it apart, so that mostly one group at a time waits for scratch; the ring then
        // holds `stride` panels per group more.)
        constexpr int PPB = 32 / SPP;                        // panels per block of up to 32 values
        const int ahead = BIG ? p.ahead + grp * p.stride / 4 : max(0, (PR - n_pl) / 4);           // own panels
        int next_blk = ahead;                                // own panel before which the next block is due
        float* rg = red + grp * (8 * kMBlkSlots);            // [block parity][4 lane quarters][kMBlkSlots]
        int c_s = 0, c_blk = 0, c_left = 0, c_par = 0;       // layer, next block, blocks left, parity of the block count
        // false: a wait of some warp of the group was abandoned, all four leave
        auto contract_block = [&]() -> bool {
            const int vg0 = c_s * n_vt, pbase = (c_s * n_pl) % PR;
            // first panel of the layer that this group scored; its others follow every fourth panel
            const int g1 = 2 * ((pair - vg0) & 1) + half;
            const int own = (n_pl - g1 + 3) / 4, b0 = c_blk * PPB;
            if (c_blk == 0) {
                bool ready = true;
                if (lane == 0) ready = mbar_wait(smem_u32(&ctl.stat_full[c_s & 1]), (c_s >> 1) & 1, abort_flag);
                if (!__shfl_sync(0xffffffffu, ready, 0)) ok = false;   // (the failed wait has raised the abort flag)
                __syncwarp();          // orders the other lanes' reads below behind the wait; a shuffle alone does not
                tmem_st_wait();
                // every record of the head is there (the statistics warp has seen the count): each thread merges those of
                // its row, straight from the L2. 18 records took the statistics warp 3 us of a layer's 16 beside four busy
                // warps (two query tiles: 8), a group's 128 threads take 0.5. With very many as well, up to 144 of one head, although each of the
                // four groups reads them all: 128 rows, 2 heads, 32 layers of 8192 tokens 454 -> 276 us, 1 head, 12000 tokens 594 -> 323.
                float M = -CUDART_INF_F, S = 0.f;
                const size_t step = static_cast<size_t>(n_mt) * 256;
                const float* src = p.cta_stat + ((static_cast<size_t>(c_s & 1) * gridDim.x + static_cast<size_t>(hkv) * p.cph) * n_mt +
                                                 (two ? pair : 0)) * 256 + row;
                constexpr int kF = BIG ? 9 : 18;         // records in flight (18 in the small form: 2048 tokens 111 -> 108 us; in the big one 42450 tokens 1174 -> 1207)
                for (int j0 = 0; ok && j0 < p.cph; j0 += kF) {
                    float rm[kF], rl[kF];
#pragma unroll
                    for (int j = 0; j < kF; ++j) {
                        const bool in = j0 + j < p.cph;
                        rm[j] = in ? __ldcg(src + (j0 + j) * step) : -CUDART_INF_F;
                        rl[j] = in ? __ldcg(src + (j0 + j) * step + 128) : 0.f;
                    }
                    float bm = M;
#pragma unroll
                    for (int j = 0; j < kF; ++j) bm = fmaxf(bm, rm[j]);
                    float acc = S * ex2_below(M, bm);
#pragma unroll
                    for (int j = 0; j < kF; ++j) acc += rl[j] * ex2_below(rm[j], bm);
                    M = bm;
                    S = acc;
                }
                gstat[grp * 256 + row] = M;                // (read back by this thread only)
                gstat[grp * 256 + 128 + row] = 1.0f / S;
            }
            const float* gm = gstat + grp * 256;
            const float mi = gm[row], li = gm[128 + row];
            float* rb = rg + c_par * (4 * kMBlkSlots);
            if (own > 0) {
                float v[32], pm[PPB];
                int slot_of[PPB];
#pragma unroll
                for (int u = 0; u < PPB; ++u) {
                    const int pl = min(g1 + 4 * (b0 + u), n_pl - 1);
                    int slot = pbase + pl;
                    slot -= (slot >= PR) ? PR : 0;
                    slot_of[u] = slot;
                }
                if constexpr (BIG) {
                    float vp[PPB * PCOLS];
#pragma unroll
                    for (int u = 0; u < PPB; ++u) {
                        if (slot_of[u] < p.ring_on) {
                            part_load<PCOLS>(lane_addr + static_cast<uint32_t>(PART0 + slot_of[u] * PCOLS), &vp[u * PCOLS]);
                        } else {
                            spill_load<PCOLS, 32>(spill + (slot_of[u] - p.ring_on) * spill_step, 32, lane, &vp[u * PCOLS], drop);
                        }
                    }
                    tmem_ld_wait();
#pragma unroll
                    for (int u = 0; u < PPB; ++u) {
                        pm[u] = vp[u * PCOLS + SPP];
#pragma unroll
                        for (int q = 0; q < SPP; ++q) v[u * SPP + q] = vp[u * PCOLS + q];
                    }
                } else {
#pragma unroll
                    for (int u = 0; u < PPB; ++u)
                        part_load<SPP>(lane_addr + static_cast<uint32_t>(PART0 + slot_of[u] * SPP), &v[u * SPP]);
                    tmem_ld_wait();
#pragma unroll
                    for (int u = 0; u < PPB; ++u) pm[u] = pmax[slot_of[u] * 128 + row];
                }
#pragma unroll
                for (int e = PPB * SPP; e < 32; ++e) v[e] = 0.f;
#pragma unroll
                for (int u = 0; u < PPB; ++u) {
                    const bool have = active && b0 + u < own;
                    const float f = have ? ex2_approx(pm[u] - mi) * li : 0.f;
#pragma unroll
                    for (int q = 0; q < SPP; ++q) v[u * SPP + q] = have ? v[u * SPP + q] * f : 0.f;
                }
                rb[quarter * kMBlkSlots + lane] = warp_transpose_reduce(v, lane);
            }
            // the block's sums are there; and a uniform decision to go on (the two halves of rg alternate: a half is written
            // again only after the next block's barrier, which its readers reach behind their reads)
            if (named_barrier_or(kBarGroup + grp, 128, !ok || ctl.abort_flag != 0)) return false;
            if (gt < min(own - b0, PPB) * SPP) {
                const int pl = g1 + 4 * (b0 + gt / SPP);
                const int kp = two ? (pl >> 2) * 2 + (pl & 1) : pl;          // panel of the key range
                const int ch = ch0 + kp * SPP + gt % SPP;
                if (ch < p.C)
                    p.scores[((static_cast<size_t>(c_s) * p.Hkv + hkv) * n_mt + (two ? pair : 0)) * p.Cpad + ch] =
                        (rb[gt] + rb[kMBlkSlots + gt]) + (rb[2 * kMBlkSlots + gt] + rb[3 * kMBlkSlots + gt]);
            }
            ++c_blk;
            c_par ^= 1;
            if (--c_left == 0) {
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctl.sc_done[c_s & 1]));      // announced by the statistics warp
            }
            return true;
        };
        bool alive = true;
        // the panels of slot s that belong to this thread's group, and the contraction of the layer before
        auto do_layer = [&](int s) {
            const int vg0 = s * n_vt, pbase = (s * n_pl) % PR;
            int done = 0;
            next_blk = ahead;
            for (int vt = (pair - vg0) & 1; vt < n_vt; vt += 2, ++done) {
                if (c_left > 0 && done >= next_blk) {
                    if (!contract_block()) { alive = false; return; }
                    if constexpr (BIG) next_blk += p.stride;
                }
                if (!ok) continue;           // (an abandoned wait: only the group's barriers are still kept)
                const int ti = two ? vt >> 1 : vt;
                const int pc = 2 * (vg0 + vt) + half;        // panel number since the start of the launch
                const int aslot = BIG ? pair : pc % kMAccSlots;
                const int use = BIG ? (vg0 + vt) >> 1 : pc / kMAccSlots;
                const int acol = BIG ? pair * kRUmmaN + half * WP : (pc % kMAccBufs) * kMAccN + half * COL1;
                if (!mbar_wait_warp(smem_u32(&ctl.tfull[aslot]), use & 1, abort_flag)) { ok = false; continue; }
                tc_fence_after();
                float v[WP];
                load_panel<WP>(lane_addr + static_cast<uint32_t>(acol), v);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&ctl.tempty[aslot]));
                const int pl = vt * 2 + half;
                int slot = pbase + pl;
                slot -= (slot >= PR) ? PR : 0;
                const int j0 = (t_begin + ti) * TILE + half * WP;
                float pr[PCOLS], m2, l;          // (big variant: the panel maximum behind the chunk sums)
                auto emit = [&](int ch, float acc) { pr[ch] = acc; };
                if (j0 + WP <= p.P)
                    panel_fast<C_STATIC, WP>(v, p.sl2, emit, &m2, &l);
                else
                    panel_static_tail<C_STATIC, WP>(v, p.sl2, emit, j0, p.P, last_visible, &m2, &l);
                if constexpr (BIG) {
                    pr[SPP] = m2;
                    if (slot < p.ring_on) {
                        part_store<PCOLS>(lane_addr + static_cast<uint32_t>(PART0 + slot * PCOLS), pr);
                    } else {
                        spill_store<PCOLS, 32>(spill + (slot - p.ring_on) * spill_step, 32, lane, pr, keep);
                    }
                } else {
                    part_store<SPP>(lane_addr + static_cast<uint32_t>(PART0 + slot * SPP), pr);
                    pmax[slot * 128 + row] = m2;
                }
                merge_ml(run_m, run_l, m2, l);
            }
        };
        // end of slot s: this group's (max, sum) per row -> shared memory. The last of the groups' warps that hold the same 32 rows
        // merges their parts and stores them; the statistics warp announces the CTA's record when all of it is there (no
        // block-wide barrier on the scoring warps' path).
        auto publish = [&](int s) {
            float* rc = rec + (s & 1) * 3072;
            rc[(grp * 2 + 0) * 128 + row] = active ? run_m : -CUDART_INF_F;
            rc[(grp * 2 + 1) * 128 + row] = active ? run_l : 0.f;
            run_m = -CUDART_INF_F;
            run_l = 0.f;
            __threadfence_block();
            __syncwarp();
            const int mt = two ? pair : 0, n_g = two ? 2 : 4;
            int* cnt = &ctl.pub_count[s & 1][mt][quarter];
            int old = 0;
            if (lane == 0) old = atomicAdd(cnt, 1);
            if (__shfl_sync(0xffffffffu, old, 0) == n_g - 1) {
                __threadfence_block();
                float M = -CUDART_INF_F, S = 0.f, m[4], l[4];
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    m[g] = g < n_g ? rc[((mt * 2 + g) * 2) * 128 + row] : -CUDART_INF_F;
                    l[g] = g < n_g ? rc[((mt * 2 + g) * 2 + 1) * 128 + row] : 0.f;
                }
                merge_records(M, S, m, l);
                float* dst = p.cta_stat + ((static_cast<size_t>(s & 1) * gridDim.x + blockIdx.x) * n_mt + mt) * 256;
                dst[row] = M;
                dst[128 + row] = S;
                __syncwarp();
                if (lane == 0) {
                    *cnt = 0;
                    mbar_arrive(smem_u32(&ctl.pub_done[s & 1]));
                }
            }
        };
        for (int s = 0; s <= p.n_compute && alive; ++s) {
            if (s < p.n_compute) do_layer(s);
            while (alive && c_left > 0) alive = contract_block();
            if (alive && s < p.n_compute) {
                publish(s);
                const int own = (n_pl - (2 * ((pair - s * n_vt) & 1) + half) + 3) / 4;
                c_s = s;
                c_blk = 0;
                c_left = max(1, (own + PPB - 1) / PPB);
            }
        }
        if (!ok && lane == 0) ctl.abort_flag = 1;
    } else if (warp == 19) {
        // ------------------------------------------------------------------ statistics warp
        // Per slot: announce the CTA's record once it is stored, wait (bounded) until every CTA of the scoring head has
        // announced its own, let the epilogue merge them, and announce the CTA's chunk scores once the epilogue has stored them.
        bool ok = true;
        for (int s = 0; s < p.n_compute && ok; ++s) {
            bool w_ok = true;
            if (lane == 0)
                w_ok = mbar_wait(smem_u32(&ctl.pub_done[s & 1]), static_cast<uint32_t>(s >> 1) & 1u, abort_flag);
            if (!__shfl_sync(0xffffffffu, w_ok, 0)) break;
            __syncwarp();
            // release, behind the wait that acquired what the epilogue warps stored: the record is visible to whoever sees the count
            if (lane == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p.cnt_a + hkv) : "memory");
            if (!wait_counter_warp(p.cnt_a + hkv, static_cast<unsigned>(s + 1) * p.cph, abort_flag)) break;
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(smem_u32(&ctl.stat_full[s & 1]));
                // the epilogue forms the slot's chunk scores next; announce them when they are stored
                if (mbar_wait(smem_u32(&ctl.sc_done[s & 1]), static_cast<uint32_t>(s >> 1) & 1u, abort_flag))
                    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p.cnt_b + hkv) : "memory");
                else
                    ok = false;
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
        }
    } else if (warp == 18) {
        // ------------------------------------------------------------------ tail: row copies
        // Once the selector CTA has published the head's kept-chunk list of a slot, this warp fetches the list and moves this
        // CTA's share of the rows - whole chunks and window pieces - through the staging slots with bulk copies, for the computed
        // layer and for every layer that reuses its indices. Rows that are not adjacent in memory (e.g. token-major caches)
        // arrive through tensor maps whose box is a chunk: one copy as well, whatever the strides.
        // The units of all these layers are one sequence; a round takes `lanes` of them, a lane each, through one of n_sets sets of
        // slots, so that a set is loaded while the others are stored. What bounds this warp is not the copies but its own instructions,
        // which wait for their turn beside 16 busy warps: one thread took 630 ns a unit, of which 60 waiting for copies (32768
        // tokens; 420 ns when nothing else ran), more than the scoring took where two layers share a list.
        uint8_t* tbase = dyn + p.off_tail;
        int* row = reinterpret_cast<int*>(tbase);            // [4 + kkpad]: n_tok, -, -, -, kept chunk ids
        const uint32_t stage0 = smem_u32(tbase + p.sel_row_bytes);
        const int* sel = row + 4;
        const int Q = p.cph, q = part;                       // CTAs of this KV head
        constexpr int kSl = C_STATIC <= 10 ? kMSlots : 0;    // staging slots where every head dim has the most
        const int n_slots = kSl ? kSl : p.copy_slots;
        const int lanes = n_slots >= 4 ? n_slots / 2 : 1, n_sets = n_slots >= 4 ? 2 : n_slots;
        const int kk = min(p.k, p.C);
        const int wu = (p.w + C_STATIC - 1) / C_STATIC;      // the window as pseudo-chunks of up to c rows
        const int U = kk + wu;                               // copy units of the head
        const int u_begin = static_cast<int>(static_cast<long long>(U) * q / Q);
        const int u_end = static_cast<int>(static_cast<long long>(U) * (q + 1) / Q);
        const int n_units = u_end - u_begin;
        const uint32_t row_bytes = static_cast<uint32_t>(p.d) * 2u;
        const uint32_t half_slot = static_cast<uint32_t>(p.stage_slot_bytes) / 2u;
        uint32_t phase = 0;                                  // parity of this lane's next wait, a bit per set
        bool ok = true;
        for (int li = 0; li < p.n_layers;) {
            const int s = p.layer[li].slot;
            int lj_end = li + 1;
            while (lj_end < p.n_layers && !p.layer[lj_end].computes) ++lj_end;
            if (lane == 0) {
                ok = wait_counter(p.cnt_c + hkv, static_cast<unsigned>(s + 1), abort_flag, 200);
                if (ok) {
                    asm volatile("fence.acq_rel.gpu;" ::: "memory");
                    const uint32_t bar = smem_u32(&ctl.sfull);
                    mbar_arrive_expect_tx(bar, static_cast<uint32_t>(p.sel_row_bytes));
                    // the list was written with ordinary stores by the selector CTA
                    asm volatile("fence.proxy.async.global;" ::: "memory");
                    bulk_load(smem_u32(row), p.sel_rows + (static_cast<size_t>(s) * p.Hkv + hkv) * (p.sel_row_bytes / 4),
                              static_cast<uint32_t>(p.sel_row_bytes), bar);
                }
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (ok) ok = mbar_wait(smem_u32(&ctl.sfull), static_cast<uint32_t>(s) & 1u, abort_flag);
            if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
            const int n_tok = row[0];
            if (lane < lanes && n_units > 0) {
                auto unit = [&](int u, int& src_row, int& dst_row, int& rows) {
                    if (u < kk) {
                        src_row = sel[u] * C_STATIC;
                        dst_row = u * C_STATIC;
                        rows = min(C_STATIC, p.P - src_row);
                    } else {
                        const int j = u - kk;
                        src_row = p.P + j * C_STATIC;
                        dst_row = n_tok + j * C_STATIC;
                        rows = min(C_STATIC, p.L - src_row);
                    }
                };
                auto issue_load = [&](int lj, int idx, int set) {
                    int sr, dr, rows;
                    unit(u_begin + idx, sr, dr, rows);
                    const uint32_t slot = static_cast<uint32_t>(set * lanes + lane);
                    const uint32_t bar = smem_u32(&ctl.gfull[slot]);
                    const uint32_t dst = stage0 + slot * p.stage_slot_bytes;
                    if (!p.strided) {
                        const ModelLayer& ly = p.layer[lj];
                        const size_t from = (static_cast<size_t>(hkv) * p.L + sr) * row_bytes;
                        const uint32_t bytes = static_cast<uint32_t>(rows) * row_bytes;
                        mbar_arrive_expect_tx(bar, 2u * bytes);
                        bulk_load(dst, reinterpret_cast<const char*>(ly.K) + from, bytes, bar);
                        bulk_load(dst + half_slot, reinterpret_cast<const char*>(ly.V) + from, bytes, bar);
                    } else {
                        // (a box is always whole: rows past the chunk's or window's end are not stored, past L they are zeros)
                        mbar_arrive_expect_tx(bar, 2u * static_cast<uint32_t>(p.copy_box_bytes));
                        tma_load_3d(dst, &p.tm_rk[lj], bar, 0, sr, hkv);
                        tma_load_3d(dst + half_slot, &p.tm_rv[lj], bar, 0, sr, hkv);
                    }
                };
                // this lane's next unit to load, and to store: (layer, unit of the CTA's share), `lanes` units apart
                int lj_l = li, ix_l = lane, lj_s = li, ix_s = lane, set = 0;
                auto next = [&](int& lj, int& ix) {
                    ix += lanes;
                    while (ix >= n_units) { ix -= n_units; ++lj; }
                };
                while (ix_l >= n_units) { ix_l -= n_units; ++lj_l; }
                lj_s = lj_l;
                ix_s = ix_l;
                for (int i = 0; i < n_sets && lj_l < lj_end; ++i) {
                    issue_load(lj_l, ix_l, i);
                    next(lj_l, ix_l);
                }
                while (lj_s < lj_end) {
                    const uint32_t slot = static_cast<uint32_t>(set * lanes + lane);
                    ok = mbar_wait(smem_u32(&ctl.gfull[slot]), phase >> set & 1u, abort_flag);
                    if (!ok) break;
                    phase ^= 1u << set;
                    int sr, dr, rows;
                    unit(u_begin + ix_s, sr, dr, rows);
                    const ModelLayer& ly = p.layer[lj_s];
                    const uint32_t bytes = static_cast<uint32_t>(rows) * row_bytes, from = stage0 + slot * p.stage_slot_bytes;
                    const size_t to = (static_cast<size_t>(hkv) * p.n_max + dr) * row_bytes;
                    bulk_store(reinterpret_cast<char*>(ly.out_K) + to, from, bytes);
                    bulk_store(reinterpret_cast<char*>(ly.out_V) + to, from + half_slot, bytes);
                    bulk_commit();
                    if (lj_l < lj_end) {
                        bulk_wait_read<0>();                 // the slot is loaded again
                        issue_load(lj_l, ix_l, set);
                        next(lj_l, ix_l);
                    }
                    next(lj_s, ix_s);
                    if (++set == n_sets) set = 0;
                }
                bulk_wait_read<0>();                         // the slots are reused by the next list's first loads
            }
            __syncwarp();                                    // (and the list itself)
            if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
            li = lj_end;
        }
        bulk_wait_all();
        if (!ok) ctl.abort_flag = 1;
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    if (threadIdx.x == 0) {
        if (ctl.abort_flag) atomicExch(p.status, 1);
        const unsigned old = atomicAdd(p.exits, 1u);
        if (old + 1u == gridDim.x) {
            for (int h = 0; h < p.Hkv; ++h) { p.cnt_a[h] = 0u; p.cnt_b[h] = 0u; p.cnt_c[h] = 0u; }
            *p.exits = 0u;
            __threadfence();
        }
    }
}

}  // namespace

// Selector CTAs: four take the SMs that eight scoring heads leave idle anyway; more of them, one a head up to 16, where that costs the
// scoring nothing (below); 0: no such choice.
constexpr int kMSelFew = 4, kMSelMany = 16;
static int many_selectors(int Hkv, int max_ctas) {
    const int n = Hkv < kMSelMany ? Hkv : kMSelMany;
    return Hkv > kMSelFew && max_ctas - n >= Hkv ? n : 0;
}

bool make_model_plan(int L, int R, int Hkv, int d, int c, int C, int k, int reuse, int max_ctas, int smem_limit, ModelPlan* plan, int n_sel) {
    // the chunk sizes that are compiled in, as in layer_resident.cu
    if (c != 5 && c != 8 && c != 10 && c != 16 && c != 20 && c != 32) return false;
    if (R < 1 || R > 256 || (d != 64 && d != 128) || L < 1 || C < 1 || k < 1 || Hkv < 1 || Hkv > kResidentMaxHeads)
        return false;
    const int kk = k < C ? k : C;
    if (kk > kSelCap || C > kSelMaxChunks) return false;     // the selector stages the kept chunk ids in shared memory
    if (max_ctas < Hkv + 1) return false;
    ModelPlan p{};
    p.c_static = c;
    p.n_mt = R > 128 ? 2 : 1;
    p.tile = 2 * panel_keys(c);
    p.spp = panel_keys(c) / c;
    p.n_tiles = (L + p.tile - 1) / p.tile;
    // What a layer takes with n selectors, ns: scoring (a chain of latencies and some 1.1 us a product of a tile), the selections of one
    // selector's heads, the copies of one CTA's units, whichever is longest; fitted to calls of 2048 to 42450 tokens. As many selectors as there are
    // if that is at most 4 % more: their lists come sooner, which shortens the end of the launch. us with four -> with one a head (16
    // at most), 10 % kept: 8 heads, 128 rows 4096 tokens x12 102.5 -> 93.5, 16000 x12 138 -> 130, 20000 x8 116 -> 108; 256 rows 16000 x12 237 -> 232;
    // 12 heads 2048 x9 99 -> 68, 16000 x6 118.5 -> 107; 16 heads 2048 140 -> 84 (x9, 4096), 32 heads 240 -> 89, 8192 297 -> 180. Where a CTA gets another
    // tile or the copies are the longest, four are better: 8 heads, 256 rows 8192 tokens x12 144 -> 154, 32768 x8 280 -> 294; 128 rows, chunks of 5,
    // a fifth kept, indices shared by two, 12000 x12 141 -> 143; 24 heads 32768 x6, a fifth kept, shared by three 298 -> 308.
    p.n_sel = Hkv < kMSelFew ? Hkv : kMSelFew;
    const int many = many_selectors(Hkv, max_ctas);
    if (many > 0) {
        auto layer_ns = [&](int n) {
            int cph = (max_ctas - n) / Hkv;
            if (cph > p.n_tiles) cph = p.n_tiles;
            const long long score = 3500 + 1100ll * p.n_mt * ((p.n_tiles + cph - 1) / cph);
            const long long select = static_cast<long long>((Hkv + n - 1) / n) * (4000 + C * 4ll / 5);
            const long long copy = static_cast<long long>(reuse) * kk * (200 + 13 * c) / cph;
            const long long longer = score > select ? score : select;
            return longer > copy ? longer : copy;
        };
        if (max_ctas - kMSelFew < Hkv || 100 * layer_ns(many) <= 104 * layer_ns(kMSelFew)) p.n_sel = many;
    }
    if (n_sel > 0) p.n_sel = n_sel;
    if (max_ctas - p.n_sel < Hkv) p.n_sel = max_ctas - Hkv;
    p.cph = (max_ctas - p.n_sel) / Hkv;
    if (p.cph > p.n_tiles) p.cph = p.n_tiles;
    p.n_score = p.cph * Hkv;
    p.grid = p.n_score + p.n_sel;
    p.t_max = (p.n_tiles + p.cph - 1) / p.cph;
    // Panels of a CTA and layer; the ring should hold them and at least kMinAhead of the next layer, whose scoring
    // hides the exchange of row statistics. Where tensor memory holds fewer the ring continues in scratch.
    constexpr int kMinAhead = 8, kBigAhead = 5;
    const int n_pl = 2 * p.n_mt * p.t_max;
    p.big = p.n_mt == 2 || n_pl + kMinAhead > model_ring_panels(c, false);
    p.ahead = p.stride = 0;
    if (p.big) {
        // per epilogue group: kBigAhead panels (about 10 us) until the statistics are there, then a block of the contraction
        // every `stride` panels so that the last one is done near the end of the layer
        const int own = (n_pl + 3) / 4, ppb = 32 / p.spp, blocks = (own + ppb - 1) / ppb;
        p.ahead = own < kBigAhead ? own : kBigAhead;
        p.stride = (own - p.ahead) / blocks;
        p.stride = p.stride < 1 ? 1 : (p.stride > ppb ? ppb : p.stride);
        p.ring_on = model_ring_panels(c, true);
        p.ring = (n_pl + 4 * (p.ahead + p.stride) + 3) / 4 * 4;
        if (p.ring < p.ring_on) p.ring = p.ring_on;
        // (`stride` falls where another block begins, and the ring with it)
        const int widest = own - p.ahead < 1 ? 1 : (own - p.ahead > ppb ? ppb : own - p.ahead);
        p.ring_reserve = (n_pl + 4 * (p.ahead + widest) + 3) / 4 * 4;
        if (p.ring_reserve < p.ring_on) p.ring_reserve = p.ring_on;
    } else {
        p.ring_on = p.ring = p.ring_reserve = model_ring_panels(c, false);
    }
    p.spill_rows = R < 128 ? (R + 31) & ~31 : 128;
    const int KB = d / 64, stage = p.tile * 128;
    const int q_bytes = p.n_mt * KB * kRQTileBytes;
    const int pmax_bytes = p.big ? 0 : p.ring * 128 * 4;     // the panel-maxima ring: one row set per ring panel
    p.copy_slots = c <= 10 ? kMSlots : model_copy_slots(c, d);
    p.stage_slot_bytes = 2 * c * d * 2;                        // K rows and V rows of one chunk
    p.sel_row_bytes = ((4 + kk) * 4 + 127) & ~127;
    const int tail_bytes = p.sel_row_bytes + p.copy_slots * p.stage_slot_bytes + 128;
    const int fixed = 1024 + q_bytes + 1024 + pmax_bytes + kMMiscBytes + tail_bytes;
    int ns = (smem_limit - 512 - fixed) / stage;               // (the control block is larger than the layer kernel's)
    if (ns > kRMaxStages) ns = kRMaxStages;
    if (ns < 2 * KB + 1) return false;
    p.n_stages = ns;
    p.off_ring = q_bytes;
    p.off_pmax = p.off_ring + ns * stage + 1024;
    p.off_misc = p.off_pmax + pmax_bytes;
    p.off_tail = p.off_misc + kMMiscBytes;
    p.smem_bytes = 1024 + p.off_tail + tail_bytes;
    // the selector CTAs use the same allocation for their scratch and (many chunks) the keys
    const size_t sel_need = (sizeof(SelectSmem) + 127) & ~size_t(127);
    if (sel_need + 1024 > static_cast<size_t>(p.smem_bytes)) return false;
    p.sel_keys_fit = (sel_need + static_cast<size_t>(C) * 4 + 1024 <= static_cast<size_t>(p.smem_bytes)) ? 1 : 0;
    *plan = p;
    return true;
}

// Scratch of a scoring CTA for the part of the ring that is not on chip: the records, and four groups' blocks for the warps
// without rows.
static size_t model_spill_floats(const ModelPlan& plan, int ring) {
    if (ring <= plan.ring_on) return 0;
    const size_t n_w = plan.spill_rows / 32;
    return ((ring - plan.ring_on) * n_w + 4 * (4 - n_w)) * (plan.spp + 1) * 32;
}

static size_t model_floats(const ModelPlan& plan, int Hkv, int C, int n_compute, int ring) {
    return static_cast<size_t>(2) * plan.grid * plan.n_mt * 256 + static_cast<size_t>(n_compute) * Hkv * plan.n_mt * ((C + 3) & ~3) +
           static_cast<size_t>(n_compute) * Hkv * (plan.sel_row_bytes / 4) + 64 +
           static_cast<size_t>(plan.n_score) * model_spill_floats(plan, ring);
}

size_t model_scratch_floats(const ModelPlan& plan, int Hkv, int C, int n_compute) {
    return model_floats(plan, Hkv, C, n_compute, plan.ring);
}

size_t model_reserve_floats(int L, int R, int Hkv, int d, int c, int C, int k, int max_ctas, int smem_limit, int n_compute) {
    // A grid with a given number of selectors never shrinks for a longer sequence, nor does its ring_reserve; either number of
    // selectors that a sequence may have is provided for.
    size_t need = 0;
    ModelPlan p;
    for (const int n : {Hkv < kMSelFew ? Hkv : kMSelFew, many_selectors(Hkv, max_ctas)})
        if (n > 0 && make_model_plan(L, R, Hkv, d, c, C, k, 1, max_ctas, smem_limit, &p, n)) {
            const size_t m = model_floats(p, Hkv, C, n_compute, p.ring_reserve);
            need = m > need ? m : need;
        }
    return need;
}

template <int C_STATIC>
static const void* model_kernel_of(bool big) {
    return big ? reinterpret_cast<const void*>(model_kernel<C_STATIC, true>) : reinterpret_cast<const void*>(model_kernel<C_STATIC, false>);
}

cudaError_t launch_model(const ModelPlan& plan, const ModelIO& io, const CUtensorMap* tm_q, const CUtensorMap* tm_k,
                         const CUtensorMap* tm_rk, const CUtensorMap* tm_rv, const ModelLayerIO* layers, int n_layers,
                         cudaStream_t stream) {
    ModelParams* pp = new ModelParams();        // too large for the host stack frame of every caller; copied at launch
    ModelParams& p = *pp;
    int n_compute = 0;
    for (int i = 0; i < n_layers; ++i) {
        ModelLayer& ly = p.layer[i];
        ly.K = static_cast<const uint4*>(layers[i].K);
        ly.V = static_cast<const uint4*>(layers[i].V);
        ly.out_K = static_cast<uint4*>(layers[i].out_K);
        ly.out_V = static_cast<uint4*>(layers[i].out_V);
        ly.out_idx = layers[i].out_idx;
        ly.computes = layers[i].computes ? 1 : 0;
        if (ly.computes) {
            p.tm_q[n_compute] = tm_q[n_compute];
            p.tm_k[n_compute] = tm_k[n_compute];
            ++n_compute;
        }
        ly.slot = n_compute - 1;
    }
    p.n_layers = n_layers;
    p.n_compute = n_compute;
    p.L = io.L; p.P = io.L - io.w; p.w = io.w; p.R = io.R; p.d = io.d; p.n_mt = plan.n_mt;
    p.sl2 = io.sl2;
    p.strided = tm_rk != nullptr ? 1 : 0;
    p.copy_box_bytes = (plan.c_static < io.L ? plan.c_static : io.L) * io.d * 2;
    if (p.strided)
        for (int i = 0; i < n_layers; ++i) { p.tm_rk[i] = tm_rk[i]; p.tm_rv[i] = tm_rv[i]; }
    p.cph = plan.cph; p.n_tiles = plan.n_tiles; p.n_stages = plan.n_stages;
    p.q_box_rows = io.R < 128 ? io.R : 128;
    p.k_box_rows = io.L < plan.tile ? io.L : plan.tile;
    p.C = io.C; p.k = io.k; p.n_max = io.n_max; p.Hkv = io.Hkv;
    p.ring_on = plan.ring_on; p.ring = plan.ring; p.spill_rows = plan.spill_rows; p.ahead = plan.ahead; p.stride = plan.stride; p.copy_slots = plan.copy_slots;
    p.Cpad = (io.C + 3) & ~3;
    p.n_score = plan.n_score; p.n_sel = plan.n_sel;
    p.sel_row_bytes = plan.sel_row_bytes; p.sel_keys_fit = plan.sel_keys_fit;
    p.off_ring = plan.off_ring; p.off_pmax = plan.off_pmax; p.off_misc = plan.off_misc; p.off_tail = plan.off_tail;
    p.stage_slot_bytes = plan.stage_slot_bytes;
    p.cta_stat = io.scratch;
    p.scores = io.scratch + static_cast<size_t>(2) * plan.grid * plan.n_mt * 256;
    p.sel_rows = reinterpret_cast<int*>(p.scores + static_cast<size_t>(n_compute) * io.Hkv * plan.n_mt * p.Cpad);   // 16-byte aligned: Cpad % 4 == 0
    p.spill = reinterpret_cast<float*>(p.sel_rows) + static_cast<size_t>(n_compute) * io.Hkv * (plan.sel_row_bytes / 4);
    p.exits = io.counters;
    p.cnt_a = io.counters + 16;
    p.cnt_b = io.counters + 16 + kResidentMaxHeads;
    p.cnt_c = io.counters + 16 + 2 * kResidentMaxHeads;
    p.status = io.status;
    const void* kern = nullptr;
    int v = 0;
    switch (plan.c_static) {
        case 5: kern = model_kernel_of<5>(plan.big); v = 0; break;
        case 8: kern = model_kernel_of<8>(plan.big); v = 1; break;
        case 10: kern = model_kernel_of<10>(plan.big); v = 2; break;
        case 16: kern = model_kernel_of<16>(plan.big); v = 3; break;
        case 20: kern = model_kernel_of<20>(plan.big); v = 4; break;
        case 32: kern = model_kernel_of<32>(plan.big); v = 5; break;
        default: break;
    }
    v += plan.big ? 6 : 0;
    static int smem_set[12][64] = {{0}};
    int dev = 0;
    cudaError_t e = kern != nullptr ? cudaGetDevice(&dev) : cudaErrorInvalidValue;
    if (e == cudaSuccess && (dev < 0 || dev >= 64 || smem_set[v][dev] < plan.smem_bytes)) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, plan.smem_bytes);
        if (e == cudaSuccess && dev >= 0 && dev < 64) smem_set[v][dev] = plan.smem_bytes;
    }
    if (e == cudaSuccess) {
        void* params[] = {&p};
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(plan.grid);
        cfg.blockDim = dim3(kMThreads);
        cfg.dynamicSmemBytes = static_cast<size_t>(plan.smem_bytes);
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;      // the CTAs of a head wait for one another: all must be resident
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelExC(&cfg, kern, params);
    }
    delete pp;
    return e;
}

}  // namespace chunkkv
