// Causal grouped-query attention of the prefill rows: row f * (Lp - 1) + t is token t of fresh
// prompt f, its keys and values are positions 0 .. t of the prompt's KV slot.
//
// Flash attention on warp-level MMAs: a CTA takes 64 tokens of a prompt for one or two heads of a
// KV head's group (a warp: 16 tokens of a head), walks the positions in blocks of 64 through two
// shared-memory stages, and keeps scores, probabilities and outputs in registers with an online
// softmax.  The output is the next GEMM's operand, a bf16 hi/lo pair.
//
// Accuracy (q, K and V are finite fp16): probabilities enter as fp16 pairs, P = hi + lo, two MMAs: 22 bits,
// and multiples of 2^-33 of the maximum (they are scaled by 2^8).  The MMAs' accumulation truncates, so a chain
// is at most 64 dims of a score or 64 positions of an output, and chains are added in fp32.  Relative
// error of the output pair against 64 bits, 33 / 255 / 2,047 tokens: 1.94e-6 / 2.17e-6 / 1.58e-6; with fp32
// products by scalar FMAs 1.94e-6 / 2.16e-6 / 1.57e-6; with one chain over all positions 2,047 tokens had
// 1.92e-6.
//
// 64 prompts x 255 tokens of the 1.5B shape (12 heads, 2 KV heads of 128), a layer: 132 us (bound by
// MMA issue and the probabilities; 124 in single chains); 1,060 us with one row per CTA and scalar products, which
// re-read every key for every token.
#pragma once
#include "device_common.cuh"

namespace sara {

constexpr int kPreTok = 64;      // tokens per tile
constexpr int kPrePos = 64;      // positions per block
constexpr float kPrePScale = 8.f;  // log2 of the probabilities' scale

struct PrefillAttnParams {
    const uint16_t *q;       // [rows][H][hd] fp16
    uint16_t *out, *out_lo;  // [rows][H][hd] bf16 hi / lo
    const uint16_t *kv;      // slot s at kv + s * slot_stride: [2][KVH][cap][hd] fp16
    int64_t slot_stride;
    int cap, H, KVH;
    const int *row_slot;     // [rows]
    const int *rows;         // device: prefill rows (fresh prompts x (Lp - 1))
    const int *Lp;           // device: prompt length
    float scale_log2;        // log2(e) / sqrt(hd)
};

constexpr size_t prefill_attn_smem(int hd) { return (size_t)2 * 2 * kPrePos * hd * 2; }

template <int HD, int HEADS>
__global__ void __launch_bounds__(128 * HEADS, 1) prefill_attn_kernel(PrefillAttnParams p) {
    constexpr int KS = HD / 16, NT = HD / 8, GR = HD / 8;  // k-steps of q.k, dim tiles, granules of a row
    constexpr int kRow = HD * 2;                           // bytes of a K / V row
    constexpr uint32_t kTile = (uint32_t)kPrePos * kRow;
    constexpr uint32_t kSw = GR < 8 ? GR - 1 : 7;          // granule swizzle: g ^ (row & kSw)
    extern __shared__ __align__(128) uint8_t pre_smem[];
    pdl_wait_prior_grids();
    pdl_allow_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int Lpre = *p.Lp - 1, n_fresh = *p.rows / Lpre;
    const int nt = (Lpre + kPreTok - 1) / kPreTok, hp = p.H / HEADS, G = p.H / p.KVH;
    const int total = n_fresh * nt * hp;
    const uint32_t sm = smem_u32(pre_smem);
#pragma unroll 1
    for (int w = blockIdx.x; w < total; w += gridDim.x) {
        // the longest tiles first
        const int hq = w % hp, rest = w / hp, f = rest % n_fresh, ti = nt - 1 - rest / n_fresh;
        const int t0 = ti * kPreTok, head = hq * HEADS + (warp >> 2), kvh = hq * HEADS / G;
        const int nkb = (min(t0 + kPreTok, Lpre) + kPrePos - 1) / kPrePos;
        const int64_t row0 = (int64_t)f * Lpre;
        const uint16_t *kbase = p.kv + p.row_slot[row0] * p.slot_stride + (int64_t)kvh * p.cap * HD;
        const uint16_t *vbase = kbase + (int64_t)p.KVH * p.cap * HD;
        auto load = [&](int kb) {  // K and V rows of block kb into stage kb & 1
            const uint32_t st = sm + (uint32_t)(kb & 1) * 2 * kTile;
#pragma unroll 4
            for (int e = threadIdx.x; e < kPrePos * GR; e += 128 * HEADS) {
                const int r = e / GR, gr = e % GR;
                const int64_t off = (int64_t)min(kb * kPrePos + r, Lpre - 1) * HD + gr * 8;
                const uint32_t dst = st + r * kRow + ((gr ^ (r & kSw)) << 4);
                cp_async16(dst, kbase + off);
                cp_async16(dst + kTile, vbase + off);
            }
            cp_async_commit();
        };
        load(0);
        const int tok0 = t0 + (warp & 3) * 16 + g, tok1 = tok0 + 8;  // this thread's two tokens
        uint32_t qf[KS][4];
        {
            const uint16_t *q0 = p.q + ((row0 + min(tok0, Lpre - 1)) * p.H + head) * HD + 2 * t;
            const uint16_t *q1 = p.q + ((row0 + min(tok1, Lpre - 1)) * p.H + head) * HD + 2 * t;
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                qf[ks][0] = *reinterpret_cast<const uint32_t *>(q0 + 16 * ks);
                qf[ks][1] = *reinterpret_cast<const uint32_t *>(q1 + 16 * ks);
                qf[ks][2] = *reinterpret_cast<const uint32_t *>(q0 + 16 * ks + 8);
                qf[ks][3] = *reinterpret_cast<const uint32_t *>(q1 + 16 * ks + 8);
            }
        }
        float o[NT][4], m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[n][e] = 0.f;
#pragma unroll 1
        for (int kb = 0; kb < nkb; ++kb) {
            if (kb + 1 < nkb) {
                load(kb + 1);
                cp_async_wait<1>();
            } else {
                cp_async_wait<0>();
            }
            __syncthreads();
            const uint32_t ks0 = sm + (uint32_t)(kb & 1) * 2 * kTile, vs0 = ks0 + kTile;
            float s[8][4];
#pragma unroll
            for (int n = 0; n < 8; n += 2) {  // positions 8 n .. 8 n + 15
                float h[2][2][4];  // [dims below / from 64][n, n + 1]
#pragma unroll
                for (int e = 0; e < 4; ++e) h[0][0][e] = h[0][1][e] = h[1][0][e] = h[1][1][e] = 0.f;
                const int r = 8 * n + (lane & 7) + ((lane >> 4) & 1) * 8;
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) {
                    uint32_t b[4];
                    ldsm_x4(ks0 + r * kRow + (((2 * ks + ((lane >> 3) & 1)) ^ (r & kSw)) << 4), b);
                    mma_f16_16816(h[ks >> 2][0], qf[ks], b[0], b[1]);
                    mma_f16_16816(h[ks >> 2][1], qf[ks], b[2], b[3]);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    s[n][e] = h[0][0][e] + h[1][0][e];
                    s[n + 1][e] = h[0][1][e] + h[1][1][e];
                }
            }
            // s[n][e]: token tok0 (e < 2) / tok1, position 64 kb + 8 n + 2 t + (e & 1)
            float mx[2] = {m[0], m[1]};
            const bool diag = (kb + 1) * kPrePos > t0;  // the causal boundary may cross this block
#pragma unroll
            for (int n = 0; n < 8; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int pos = kb * kPrePos + 8 * n + 2 * t + (e & 1);
                    s[n][e] = !diag || pos <= (e < 2 ? tok0 : tok1) ? s[n][e] * p.scale_log2 : -INFINITY;
                    mx[e >> 1] = fmaxf(mx[e >> 1], s[n][e]);
                }
#pragma unroll
            for (int q = 0; q < 2; ++q) {  // (block 0 holds position 0, so the maxima are finite)
                mx[q] = fmaxf(mx[q], __shfl_xor_sync(0xffffffffu, mx[q], 1));
                mx[q] = fmaxf(mx[q], __shfl_xor_sync(0xffffffffu, mx[q], 2));
                const float alpha = exp2f(m[q] - mx[q]);
                m[q] = mx[q];
                l[q] *= alpha;
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    o[n][2 * q] *= alpha;
                    o[n][2 * q + 1] *= alpha;
                }
            }
            uint32_t hi[4][4], lo[4][4];  // positions 16 kk .. + 15 of the block
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
#pragma unroll
                for (int a = 0; a < 4; ++a) {  // A fragment: rows g, g + 8, g, g + 8; positions 2t.., 2t.., 8 + 2t..
                    const int n = 2 * kk + (a >> 1), q = a & 1;
                    const float p0 = exp2f(s[n][2 * q] - m[q] + kPrePScale), p1 = exp2f(s[n][2 * q + 1] - m[q] + kPrePScale);
                    l[q] += p0 + p1;
                    hi[kk][a] = pack_half2(p0, p1);
                    const __half2 h = *reinterpret_cast<const __half2 *>(&hi[kk][a]);
                    lo[kk][a] = pack_half2(p0 - __low2float(h), p1 - __high2float(h));
                }
#pragma unroll
            for (int n = 0; n < NT; n += 2) {  // the block's products in accumulators of their own, then one fp32 sum
                float d[2][4];
#pragma unroll
                for (int e = 0; e < 4; ++e) d[0][e] = d[1][e] = 0.f;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const int r = 16 * kk + (lane & 15);
                    uint32_t b[4];
                    ldsm_x4_trans(vs0 + r * kRow + (((n + (lane >> 4)) ^ (r & kSw)) << 4), b);
                    mma_f16_16816(d[0], lo[kk], b[0], b[1]);
                    mma_f16_16816(d[1], lo[kk], b[2], b[3]);
                    mma_f16_16816(d[0], hi[kk], b[0], b[1]);
                    mma_f16_16816(d[1], hi[kk], b[2], b[3]);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    o[n][e] += d[0][e];
                    o[n + 1][e] += d[1][e];
                }
            }
            __syncthreads();  // the stage is free for block kb + 2
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            l[q] += __shfl_xor_sync(0xffffffffu, l[q], 1);
            l[q] += __shfl_xor_sync(0xffffffffu, l[q], 2);
            const int tok = q ? tok1 : tok0;
            if (tok < Lpre) {
                const int64_t base = ((row0 + tok) * p.H + head) * HD + 2 * t;
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    uint16_t h0, l0, h1, l1;
                    split_bf16(o[n][2 * q] / l[q], h0, l0);
                    split_bf16(o[n][2 * q + 1] / l[q], h1, l1);
                    *reinterpret_cast<uint32_t *>(p.out + base + 8 * n) = (uint32_t)h0 | ((uint32_t)h1 << 16);
                    *reinterpret_cast<uint32_t *>(p.out_lo + base + 8 * n) = (uint32_t)l0 | ((uint32_t)l1 << 16);
                }
            }
        }
    }
}

}  // namespace sara
