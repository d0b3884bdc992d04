// Grouped-query attention of single query rows over their own KV histories, as a call of its own:
//     out[r, h] = softmax(q[r, h] . K[0..ctx_r)^T / sqrt(hd)) V[0..ctx_r)
// One cluster of up to 8 CTAs per (row, KV head) shares the row's positions; a warp takes 16 of
// them at a time.  Bound by the latency of reading K and V once: all of a step's loads (16 bytes
// a lane) go straight to registers, in the order in which the warp-level MMAs want them.
//   - Scores: A = q (row g of 8: query head g of the group), B = K^T.  Lane (g, t) loads dims
//     32 j + 8 t .. + 7 of a position, and the same dims of its head, so the order of the dims
//     inside a k-step does not matter and no fragment needs rearranging.
//   - Output: A = P, straight from the score accumulators, B = V, whose 8 x 8 blocks movmatrix
//     transposes.  Probabilities enter as fp16 pairs, P = hi + lo, two MMAs: 22 bits, and multiples of
//     2^-33 of the maximum (they are scaled by 2^8).  Against 64 bits the results are as far off as
//     with fp32 probabilities (their rounding to bf16); infinite values of V are not: 0 for a small
//     probability, times infinity.  A warp whose sums are not all finite takes them again in fp32.
// Online softmax per warp; the warps' states meet in shared memory, the CTAs' in distributed
// shared memory (no workspace, no counters, so no work list from the host either).  26 ragged rows
// of median context 758, 12 heads / 2 KV heads of 128, whole call with its synchronisation: 45 to 50 us (kernel 18,
// caches cold); 89 to 97 us with scalar products over a work list that the host built from the copied contexts.
#pragma once
#include "device_common.cuh"
#include "host_util.h"

namespace sara {

constexpr int kSplitThreads = 128;
constexpr int kSplitWarps = kSplitThreads / 32;
constexpr int kSplitMaxCtas = 8;
constexpr float kSplitPScale = 8.f;  // log2 of the probabilities' scale

struct AttnSplitParams {
    const uint16_t *q;   // [b][H][hd] fp16
    const uint16_t *kv;  // sequence i at kv + i * kv_stride: [2][KVH][cap][hd] fp16
    const int *ctx;      // [b]
    uint16_t *out;       // [b][H][hd] bf16
    int *bad;            // whether a row's ctx is out of range: then nothing is written
    int64_t kv_stride;
    int H, KVH, cap, max_ctx;
    float scale_log2;
};

// The verdict on the rows' contexts.  A kernel of its own, so that every row's counts before the first
// result is written; the attention runs beside it and waits for it only there.
static __global__ void __launch_bounds__(1024) attn_ctx_check_kernel(const int *ctx, int b, int max_ctx, int *bad) {
    pdl_allow_dependents();
    bool any = false;
    for (int i = threadIdx.x; i < b; i += blockDim.x) any = any || ctx[i] < 1 || ctx[i] > max_ctx;
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) *bad = any ? 1 : 0;
}

template <int HD>
__global__ void __launch_bounds__(kSplitThreads) attn_split_kernel(AttnSplitParams p) {
    constexpr int NJ = HD / 32;  // 16-byte loads per lane and row
    __shared__ float s_m[kSplitWarps][8], s_l[kSplitWarps][8];
    __shared__ __align__(16) float s_o[kSplitWarps][8][HD];
    __shared__ float c_m[8], c_l[8], c_o[8 * HD];  // this CTA's state, read by the cluster
    const int kvh = blockIdx.y, row = blockIdx.z, rank = (int)cluster_rank(), S = (int)gridDim.x;
    const int G = p.H / p.KVH;
    const int ctx = p.ctx[row];
    if (ctx < 1 || ctx > p.max_ctx) return;  // (every CTA of the cluster has the same row)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    uint4 q[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j)
        q[j] = g < G ? __ldg(reinterpret_cast<const uint4 *>(p.q + ((int64_t)row * p.H + kvh * G + g) * HD + 32 * j + 8 * t))
                     : make_uint4(0, 0, 0, 0);
    const uint16_t *kb = p.kv + row * p.kv_stride + (int64_t)kvh * p.cap * HD + 8 * t;
    const uint16_t *vb = kb + (int64_t)p.KVH * p.cap * HD;
    const int nblk = (ctx + 15) >> 4, b0 = rank * nblk / S, b1 = (rank + 1) * nblk / S;
    float m = -INFINITY, l = 0.f, o[NJ][4][4];
#pragma unroll
    for (int j = 0; j < NJ; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[j][i][e] = 0.f;
    // K rows of step b, and its scores: s[h][e], e < 2: head g, position 16 b + 8 h + 2 t + e
    auto load = [&](int b, int h, const uint16_t *base, uint4 (&r)[NJ]) {
        const int64_t off = (int64_t)min(b * 16 + 8 * h + g, ctx - 1) * HD;
#pragma unroll
        for (int j = 0; j < NJ; ++j) r[j] = __ldg(reinterpret_cast<const uint4 *>(base + off + 32 * j));
    };
    auto scores = [&](int b, const uint4 (&kr)[2][NJ], float (&s)[2][4]) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int e = 0; e < 4; ++e) s[h][e] = 0.f;
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const uint32_t a0[4] = {q[j].x, 0u, q[j].y, 0u}, a1[4] = {q[j].z, 0u, q[j].w, 0u};
                mma_f16_16816(s[h], a0, kr[h][j].x, kr[h][j].y);
                mma_f16_16816(s[h], a1, kr[h][j].z, kr[h][j].w);
            }
#pragma unroll
            for (int e = 0; e < 2; ++e)
                s[h][e] = b * 16 + 8 * h + 2 * t + e < ctx ? s[h][e] * p.scale_log2 : -INFINITY;
        }
    };
#pragma unroll 1
    for (int b = b0 + warp; b < b1; b += kSplitWarps) {
        uint4 kr[2][NJ], vr[2][NJ];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            load(b, h, kb, kr[h]);
            load(b, h, vb, vr[h]);
            if (b * 16 + 8 * h + g >= ctx) {  // (its probability is 0)
#pragma unroll
                for (int j = 0; j < NJ; ++j) vr[h][j] = make_uint4(0, 0, 0, 0);
            }
        }
        float s[2][4];
        scores(b, kr, s);
        float mx = m;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int e = 0; e < 2; ++e) mx = fmaxf(mx, s[h][e]);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float mr = mx == -INFINITY ? 0.f : mx;  // (every score so far is -inf: weights 0)
        const float alpha = exp2f(m - mr);
        m = mx;
        l *= alpha;
        uint32_t hi[4] = {0u, 0u, 0u, 0u}, lo[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float p0 = exp2f(s[h][0] - mr + kSplitPScale), p1 = exp2f(s[h][1] - mr + kSplitPScale);
            l += p0 + p1;
            hi[2 * h] = pack_half2(p0, p1);
            const __half2 hh = *reinterpret_cast<const __half2 *>(&hi[2 * h]);
            lo[2 * h] = pack_half2(p0 - __low2float(hh), p1 - __high2float(hh));
        }
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const uint32_t v0[4] = {vr[0][j].x, vr[0][j].y, vr[0][j].z, vr[0][j].w};
            const uint32_t v1[4] = {vr[1][j].x, vr[1][j].y, vr[1][j].z, vr[1][j].w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t w0 = movmatrix_trans(v0[i]), w1 = movmatrix_trans(v1[i]);
                o[j][i][0] *= alpha;
                o[j][i][1] *= alpha;
                mma_f16_16816(o[j][i], hi, w0, w1);
                mma_f16_16816(o[j][i], lo, w0, w1);
            }
        }
    }
    bool fin = true;
#pragma unroll
    for (int j = 0; j < NJ; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) fin = fin && isfinite(o[j][i][0]) && isfinite(o[j][i][1]);
    fin = __all_sync(0xffffffffu, fin);
    if (!fin) {
        // the warp's sums of P V once more, in fp32: each step's probabilities against the final maximum by way
        // of the room of the sums (head, position), dims NJ lane .. of every head in this lane
        float acc[8][NJ];
#pragma unroll
        for (int h = 0; h < 8; ++h)
#pragma unroll
            for (int i = 0; i < NJ; ++i) acc[h][i] = 0.f;
        const float mr = m == -INFINITY ? 0.f : m;
#pragma unroll 1
        for (int b = b0 + warp; b < b1; b += kSplitWarps) {
            uint4 kr[2][NJ];
            load(b, 0, kb, kr[0]);
            load(b, 1, kb, kr[1]);
            float s[2][4];
            scores(b, kr, s);
            __syncwarp();
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 2; ++e) s_o[warp][g][8 * h + 2 * t + e] = exp2f(s[h][e] - mr + kSplitPScale);
            __syncwarp();
#pragma unroll 1
            for (int x = 0; x < min(16, ctx - 16 * b); ++x) {
                const uint16_t *v = vb - 8 * t + (int64_t)(16 * b + x) * HD + NJ * lane;
                float f[NJ];
#pragma unroll
                for (int i = 0; i < NJ; ++i) f[i] = __half2float(__ushort_as_half(__ldg(v + i)));
#pragma unroll
                for (int h = 0; h < 8; ++h)
#pragma unroll
                    for (int i = 0; i < NJ; ++i) acc[h][i] = fmaf(s_o[warp][h][x], f[i], acc[h][i]);
            }
        }
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 8; ++h)
#pragma unroll
            for (int i = 0; i < NJ; ++i) s_o[warp][h][NJ * lane + i] = acc[h][i];
    }
    // o[j][i][e], e < 2: head g, dim 32 j + 8 t + 2 i + e
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
    if (t == 0) { s_m[warp][g] = m; s_l[warp][g] = l; }
#pragma unroll
    for (int j = 0; j < NJ && fin; ++j) {
        float4 *dst = reinterpret_cast<float4 *>(&s_o[warp][g][32 * j + 8 * t]);
        dst[0] = make_float4(o[j][0][0], o[j][0][1], o[j][1][0], o[j][1][1]);
        dst[1] = make_float4(o[j][2][0], o[j][2][1], o[j][3][0], o[j][3][1]);
    }
    __syncthreads();
    pdl_wait_prior_grids();
    if (*reinterpret_cast<volatile int *>(p.bad)) return;
    const int per = G * HD;
    for (int e = threadIdx.x; e < per; e += kSplitThreads) {
        const int h = e / HD, dd = e % HD;
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < kSplitWarps; ++w) M = fmaxf(M, s_m[w][h]);
        float L = 0.f, acc = 0.f;
#pragma unroll
        for (int w = 0; w < kSplitWarps; ++w) {
            const float wt = s_m[w][h] == -INFINITY ? 0.f : exp2f(s_m[w][h] - M);
            if (s_m[w][h] != -INFINITY) {
                L += wt * s_l[w][h];
                acc += wt * s_o[w][h][dd];
            }
        }
        if (S == 1) {
            p.out[((int64_t)row * p.H + kvh * G) * HD + e] = f32_to_bf16(acc / L);
        } else {
            c_o[e] = acc;
            if (dd == 0) { c_m[h] = M; c_l[h] = L; }
        }
    }
    if (S == 1) return;
    cluster_sync();
    for (int e = rank * kSplitThreads + threadIdx.x; e < per; e += S * kSplitThreads) {
        const int h = e / HD;
        float ms[kSplitMaxCtas], ls[kSplitMaxCtas], os[kSplitMaxCtas], M = -INFINITY;
#pragma unroll
        for (int c = 0; c < kSplitMaxCtas; ++c) {
            ms[c] = c < S ? ld_cluster_f32(cluster_addr(&c_m[h], c)) : -INFINITY;
            ls[c] = c < S ? ld_cluster_f32(cluster_addr(&c_l[h], c)) : 0.f;
            os[c] = c < S ? ld_cluster_f32(cluster_addr(&c_o[e], c)) : 0.f;
            M = fmaxf(M, ms[c]);
        }
        float L = 0.f, acc = 0.f;
#pragma unroll
        for (int c = 0; c < kSplitMaxCtas; ++c)
            if (ms[c] != -INFINITY) {
                const float wt = exp2f(ms[c] - M);
                L += wt * ls[c];
                acc += wt * os[c];
            }
        p.out[((int64_t)row * p.H + kvh * G) * HD + e] = f32_to_bf16(acc / L);
    }
    cluster_sync();  // no CTA leaves while its state is read
}

// The split doubles while a CTA would still hold more than 64 positions of the longest context and
// the CTAs do not yet fill the SMs several times.  16-byte aligned q, kv (and kv_stride % 8 == 0).
inline void launch_attn_split(cudaStream_t s, int sms, int b, int hd, const AttnSplitParams &p) {
    int split = 1;
    while (split < kSplitMaxCtas && p.max_ctx > 64 * split && (int64_t)b * p.KVH * split < 4 * sms) split *= 2;
    attn_ctx_check_kernel<<<1, 1024, 0, s>>>(p.ctx, b, p.max_ctx, p.bad);
    CK(cudaGetLastError());
    const dim3 grid((unsigned)split, (unsigned)p.KVH, (unsigned)b);
    if (hd == 32) launch_cluster(s, true, grid, dim3(kSplitThreads), 0, (unsigned)split, attn_split_kernel<32>, p);
    else if (hd == 64) launch_cluster(s, true, grid, dim3(kSplitThreads), 0, (unsigned)split, attn_split_kernel<64>, p);
    else launch_cluster(s, true, grid, dim3(kSplitThreads), 0, (unsigned)split, attn_split_kernel<128>, p);
}

}  // namespace sara
