// Kernel-level entry points of include/sara.h on caller-provided device buffers: the projection
// GEMM of up to 128 rows, attention of single query rows, and the Gumbel-max sampler.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <string>
#include <vector>

#include "../../include/sara.h"
#include "attention.cuh"
#include "attn_split.cuh"
#include "gemm_rows.cuh"
#include "host_util.h"
#include "step_kernels.cuh"

using namespace sara;

namespace sara {
int gemm_rows_sms() {
    constexpr int kMaxDevices = 64;
    static std::atomic<int> known[kMaxDevices];  // SMs of devices whose kernel attribute is set, 0: not yet
    int dev = 0, sms = 0;
    CK(cudaGetDevice(&dev));
    if (dev >= 0 && dev < kMaxDevices && (sms = known[dev].load(std::memory_order_acquire)) > 0) return sms;
    CK(cudaFuncSetAttribute(gemm_rows_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + kRowsRing));
    CK(cudaFuncSetAttribute(gemm_rows_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + kRowsRing));
    CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (dev >= 0 && dev < kMaxDevices) known[dev].store(sms, std::memory_order_release);
    return sms;
}
}  // namespace sara

namespace {

int sm_count() {
    int dev = 0, sms = 0;
    CK(cudaGetDevice(&dev));
    CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    return sms;
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// The workspace of the GEMM's contract (the kernel no longer uses it; sizes unchanged).
struct GemmWs {
    size_t part_bytes, cnt_bytes;
};
GemmWs gemm_ws_layout(int Nout, int sms) {
    GemmWs w;
    w.part_bytes = align_up((size_t)sms * kRowsMax * kRowsTileM * sizeof(unsigned long long), 256);
    w.cnt_bytes = align_up((size_t)(Nout / kRowsTileM) * sizeof(int), 256);
    return w;
}

template <int HD>
void launch_g(dim3 grid, int G, cudaStream_t s, const AttnParams &a) {
    switch (G) {
        case 1: attn_rows_kernel<HD, 1><<<grid, kAttnThreads, 0, s>>>(a); break;
        case 2: attn_rows_kernel<HD, 2><<<grid, kAttnThreads, 0, s>>>(a); break;
        case 4: attn_rows_kernel<HD, 4><<<grid, kAttnThreads, 0, s>>>(a); break;
        case 6: attn_rows_kernel<HD, 6><<<grid, kAttnThreads, 0, s>>>(a); break;
        default: attn_rows_kernel<HD, 8><<<grid, kAttnThreads, 0, s>>>(a); break;
    }
}

template <typename F>
int op_guard(F fn) {
    try {
        fn();
        return SARA_OK;
    } catch (const SaraError &e) {
        return e.code;
    } catch (...) {
        return SARA_EDEVICE;
    }
}

}  // namespace

extern "C" {

size_t sara_gemm_workspace_bytes(int32_t R, int32_t Nout, int32_t K) {
    (void)R;
    (void)K;
    if (Nout <= 0) return 0;
    int sms = 0;
    try {
        sms = sm_count();
    } catch (...) {
        return 0;
    }
    const GemmWs w = gemm_ws_layout(Nout, sms);
    return w.part_bytes + w.cnt_bytes;
}

int sara_gemm_bf16(const uint16_t *X, const uint16_t *W, float *Y, int32_t R, int32_t Nout, int32_t K, void *workspace,
                   size_t workspace_bytes, void *stream) {
    if (!X || !W || !Y || !workspace) return SARA_EINVAL;
    if (R < 1 || R > kRowsMax || Nout < kRowsTileM || Nout % kRowsTileM || K < kRowsTileK || K % kRowsTileK) return SARA_EINVAL;
    if ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(W)) & 15) return SARA_EINVAL;
    return op_guard([&] {
        const int sms = gemm_rows_sms();
        const GemmWs w = gemm_ws_layout(Nout, sms);
        if (workspace_bytes < w.part_bytes + w.cnt_bytes) throw SaraError(SARA_EINVAL, "workspace too small");
        launch_gemm_rows(static_cast<cudaStream_t>(stream), sms, X, W, Y, R, Nout, K);
    });
}

int sara_gemm_bf16_static(const uint16_t *X, const uint16_t *W, float *Y, int32_t R, int32_t Nout, int32_t K,
                          void *stream) {
    constexpr int kStaticMaxNout = 262144;
    if (!X || !W || !Y) return SARA_EINVAL;
    if (R < 1 || R > kRowsMax || Nout < kRowsTileM || Nout % kRowsTileM || K < kRowsTileK || K % kRowsTileK) return SARA_EINVAL;
    if (Nout > kStaticMaxNout) return SARA_EINVAL;
    if ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(W)) & 15) return SARA_EINVAL;
    return op_guard([&] { launch_gemm_rows(static_cast<cudaStream_t>(stream), gemm_rows_sms(), X, W, Y, R, Nout, K); });
}

size_t sara_attention_workspace_bytes(int32_t b, int32_t n_heads, int32_t head_dim, int32_t max_ctx) {
    if (b < 1 || n_heads < 1 || head_dim < 1 || max_ctx < 1) return 0;
    const size_t splits = (size_t)(max_ctx + 127) / 128;
    const size_t items = (size_t)b * splits;
    // partials (<= items * n_heads * (hd + 2) floats), counters [b][n_kv], items, 3 row arrays
    return align_up(items * n_heads * (head_dim + 2) * sizeof(float), 256) +
           align_up((size_t)b * n_heads * sizeof(int), 256) + align_up(items * sizeof(int2), 256) +
           align_up((size_t)b * sizeof(int) * 3, 256);
}

int sara_attention_decode(const uint16_t *q, const uint16_t *kv, int64_t kv_stride, const int32_t *ctx, uint16_t *out,
                          int32_t b, int32_t n_heads, int32_t n_kv_heads, int32_t head_dim, int32_t cap,
                          int32_t max_ctx, void *workspace, size_t workspace_bytes, void *stream) {
    if (!q || !kv || !ctx || !out || !workspace) return SARA_EINVAL;
    if (b < 1 || n_kv_heads < 1 || n_heads % n_kv_heads || n_heads / n_kv_heads > kAttnMaxG) return SARA_EINVAL;
    if (head_dim != 32 && head_dim != 64 && head_dim != 128) return SARA_EINVAL;
    if (max_ctx < 1 || max_ctx > cap || (max_ctx + 127) / 128 > kAttnMaxSplits) return SARA_EINVAL;
    // a row is read in loads of head_dim / 16 elements at least
    if (((reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(kv)) & (head_dim / 8 - 1)) ||
        (b > 1 && kv_stride % (head_dim / 16)))
        return SARA_EINVAL;
    return op_guard([&] {
        if (workspace_bytes < sara_attention_workspace_bytes(b, n_heads, head_dim, max_ctx))
            throw SaraError(SARA_EINVAL, "workspace too small");
        cudaStream_t s = static_cast<cudaStream_t>(stream);
        const int G = n_heads / n_kv_heads;
        if (G != 1 && G != 2 && G != 4 && G != 6 && G != 8) throw SaraError(SARA_EINVAL, "query group must be 1, 2, 4, 6 or 8");
        const int sms = sm_count();
        // 16-byte loads of K, V and q rows (head dims below 128 may come less aligned); the grid's
        // z and y dimensions hold 65,535 rows and KV heads
        const bool wide = ((reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(kv)) & 15) == 0 && kv_stride % 8 == 0;
        if (wide && b <= 65535 && n_kv_heads <= 65535) {
            AttnSplitParams a{};
            a.q = q;
            a.kv = kv;
            a.ctx = ctx;
            a.out = out;
            a.bad = reinterpret_cast<int *>(workspace);
            a.kv_stride = kv_stride;
            a.H = n_heads;
            a.KVH = n_kv_heads;
            a.cap = cap;
            a.max_ctx = max_ctx;
            a.scale_log2 = (float)(1.4426950408889634 / std::sqrt((double)head_dim));
            launch_attn_split(s, sms, b, head_dim, a);
            int bad = 0;
            CK(cudaMemcpyAsync(&bad, a.bad, sizeof(int), cudaMemcpyDeviceToHost, s));
            CK(cudaStreamSynchronize(s));
            if (bad) throw SaraError(SARA_EINVAL, "ctx out of range");
            return;
        }
        const size_t splits = (size_t)(max_ctx + 127) / 128;
        const size_t items_cap = (size_t)b * splits;
        uint8_t *ws = reinterpret_cast<uint8_t *>(workspace);
        float *part = reinterpret_cast<float *>(ws);
        ws += align_up(items_cap * n_heads * (head_dim + 2) * sizeof(float), 256);
        int *cnt = reinterpret_cast<int *>(ws);
        ws += align_up((size_t)b * n_heads * sizeof(int), 256);
        int2 *items = reinterpret_cast<int2 *>(ws);
        ws += align_up(items_cap * sizeof(int2), 256);
        int *row_pos = reinterpret_cast<int *>(ws);
        int *row_item0 = row_pos + b;
        int *row_slot = row_item0 + b;  // row i reads KV slot i
        // work items (row, split) from the context lengths, built on the host
        std::vector<int> hctx(b), hpos(b), hi0(b), slots(b);
        CK(cudaMemcpyAsync(hctx.data(), ctx, b * sizeof(int), cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        std::vector<int2> hitems;
        for (int i = 0; i < b; ++i) {
            if (hctx[i] < 1 || hctx[i] > max_ctx) throw SaraError(SARA_EINVAL, "ctx out of range");
            hpos[i] = hctx[i] - 1;
            hi0[i] = (int)hitems.size();
            slots[i] = i;
            for (int sp = 0; sp < (hctx[i] + 127) / 128; ++sp) hitems.push_back(make_int2(i, sp));
        }
        CK(cudaMemcpyAsync(items, hitems.data(), hitems.size() * sizeof(int2), cudaMemcpyHostToDevice, s));
        CK(cudaMemcpyAsync(row_pos, hpos.data(), b * sizeof(int), cudaMemcpyHostToDevice, s));
        CK(cudaMemcpyAsync(row_item0, hi0.data(), b * sizeof(int), cudaMemcpyHostToDevice, s));
        CK(cudaMemcpyAsync(row_slot, slots.data(), b * sizeof(int), cudaMemcpyHostToDevice, s));
        AttnParams a{};
        a.q = q;
        a.out = out;
        a.kv = kv;
        a.slot_stride = kv_stride;
        a.cap = cap;
        a.row_slot = row_slot;
        a.row_pos = row_pos;
        a.items = items;
        a.n_items = (int)hitems.size();
        a.row_item0 = row_item0;
        a.n_heads = n_heads;
        a.n_kv = n_kv_heads;
        a.chunk = 128;
        a.scale_log2 = (float)(1.4426950408889634 / std::sqrt((double)head_dim));
        a.part = part;
        a.cnt = cnt;
        CK(cudaMemsetAsync(cnt, 0, (size_t)b * n_heads * sizeof(int), s));
        dim3 grid(std::max(1, sms * 4 / n_kv_heads), n_kv_heads);
        if (head_dim == 32) launch_g<32>(grid, G, s, a);
        else if (head_dim == 64) launch_g<64>(grid, G, s, a);
        else launch_g<128>(grid, G, s, a);
        CK(cudaGetLastError());
        CK(cudaStreamSynchronize(s));  // the host vectors above back in-flight copies
    });
}

int sara_sample(const float *logits, int32_t R, int32_t V, uint64_t sample_seed, const int64_t *uid, const int32_t *t,
                int32_t *token, void *stream) {
    if (!logits || !uid || !t || !token || R < 1 || V < 1) return SARA_EINVAL;
    return op_guard([&] {
        cudaStream_t s = static_cast<cudaStream_t>(stream);
        if (V <= kSampleShort) {
            sample_short_rows_kernel<<<R, 256, 0, s>>>(logits, V, sample_seed, uid, t, token);
            CK(cudaGetLastError());
            return;
        }
        const int ctas = sample_ctas(R, V, sm_count());
        launch_cluster(s, false, dim3((unsigned)R * ctas), dim3(256), 0, ctas,
                       sample_rows_kernel, logits, (int)V, sample_seed, uid, t, (int *)token, ctas);
    });
}

}  // extern "C"
