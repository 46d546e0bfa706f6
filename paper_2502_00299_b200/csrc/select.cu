// Stand-alone top-k chunk selection kernel: one CTA per KV head (see select.cuh).
#include "internal.h"
#include "select.cuh"

namespace chunkkv {

namespace {

constexpr int kSelThreads = 512;

constexpr size_t kSelBytes = (sizeof(SelectSmem) + 127) & ~size_t(127);

// Dynamic shared memory: kSelBytes, then key_bytes for the keys where select_kept does not hold them in registers (they are
// recomputed from the scores on every use if key_bytes is 0). staged: the kept ids fit the staging buffer of select_kept.
__global__ void __launch_bounds__(kSelThreads)
select_kernel(const float* __restrict__ scores, int L, int w, int c, int C, int k, int n_max,
              int32_t* __restrict__ out_idx, int key_bytes, bool staged, int tok_cap) {
    extern __shared__ __align__(128) uint8_t smem_raw[];      // (SelectSmem is read 16 bytes at a time)
    SelectSmem& sm = *reinterpret_cast<SelectSmem*>(smem_raw);
    uint32_t* kbuf = reinterpret_cast<uint32_t*>(smem_raw + kSelBytes);
    const int h = blockIdx.x;
    const float* sc = scores + static_cast<size_t>(h) * C;
    int32_t* out = out_idx + static_cast<size_t>(h) * n_max;
    if (staged && (key_bytes > 0 || C <= kSelThreads * select_reg_keys(kSelAlone)))
        select_head<kSelAlone>(sc, nullptr, L, w, c, C, k, n_max, out, sm, kbuf, tok_cap);
    else
        select_head_rows(sc, nullptr, L, w, c, C, k, n_max, out, sm, key_bytes > 0 ? kbuf : nullptr, tok_cap);
}

}  // namespace

cudaError_t launch_select(const float* scores, int L, int Hkv, int w, int c, int C, int k, int n_max,
                          int32_t* out_idx, cudaStream_t stream, int tok_cap) {
    // thousands of chunks per head: eight CTAs per head
    if (select_cluster_applies(C, k)) return launch_select_cluster(scores, L, Hkv, w, c, C, k, n_max, out_idx, stream, tok_cap);
    const bool staged = (k < C ? k : C) <= kSelCap && C <= kSelMaxChunks;
    if (staged && C <= kSelThreads * select_reg_keys(kSelAlone)) {
        select_kernel<<<Hkv, kSelThreads, kSelBytes, stream>>>(scores, L, w, c, C, k, n_max, out_idx, 0, true, tok_cap);
        return cudaGetLastError();
    }
    // more: the keys of a head live in dynamic shared memory if they fit behind the selection scratch
    // (beyond the 48 KB every kernel may use, so the kernel opts in), else they are recomputed
    const size_t want = static_cast<size_t>(C) * 4;
    int key_bytes = 0, dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const long room = static_cast<long>(optin) - static_cast<long>(kSelBytes) - 1024;
    if (room > 0 && want <= static_cast<size_t>(room)) {
        if (cudaFuncSetAttribute(select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(room + kSelBytes)) == cudaSuccess)
            key_bytes = static_cast<int>(want);
        else
            cudaGetLastError();
    }
    select_kernel<<<Hkv, kSelThreads, kSelBytes + key_bytes, stream>>>(scores, L, w, c, C, k, n_max, out_idx, key_bytes, staged, tok_cap);
    return cudaGetLastError();
}

}  // namespace chunkkv
