// Projection GEMM of the prefill (except at a few rows: see kPrefillFewRows):
//     Y[r][n] = sum_c (X_hi[r][c] + X_lo[r][c]) * W[n][c]
// (two MMAs per weight element and row: the activation is a bf16 hi/lo pair).  128 rows are the MMA's M, 256
// features its N, hi and lo accumulate into one accumulator, so a stage of 64 KB (32 KB of weights, 16 KB each of
// hi and lo) feeds eight N = 256 MMAs of ~130 cycles: 61 bytes a cycle, where 128 x 128 tiles need 86.  Three
// stages; two accumulators, so that the epilogue of a tile overlaps the next one's MMAs; the
// thread that finishes a row holds 128 of its features, so rotation pairs, gate and up, and the
// sums of squares of 128 features need no exchange.
// Bound by operand traffic: gate/up of 16,320 rows (1.5B shape) takes 1.27 ms, 1.41 PFLOP/s, with the tensor pipe
// 63 % busy and DRAM 73 %: 6.75 of the 14.2 GB that the SMs load come from DRAM, since the CTAs walk the 55 MB of
// weights out of step while the results pass through L2.
//
// Work split: stream-K.  The (tile, chunk) units are cut into gridDim.x equal contiguous ranges.
// A tile that spans CTAs is summed from fp32 partial tiles in CTA order by the CTA that arrives
// last (a counter per tile, nobody waits): the sums do not depend on the order of arrival.
//
// Warp roles (320 threads): warp 0 producer, warp 1 MMA issuer and tensor-memory owner, warps 2..9
// epilogue (warp w: tensor-memory lanes 32 (w % 4) .., columns 128 ((w - 2) / 4) ..).
#pragma once
#include "device_common.cuh"
#include "gemm_tc.cuh"

namespace sara {

// Up to kPrefillFewRows rows a model with long reductions (more than kPrefillFewChunks chunks) runs the
// few-row GEMM (gemm_tc.cuh) instead: there the finishing CTA's sum of the contributors' partial
// tiles weighs more than the units.  A 5-layer prefill and decode step, few-row / this kernel, ms:
// 1.5B shape, 32 rows 0.79 / 0.94, 48 rows 0.92 / 0.96, 64 rows 0.95 / 0.98, 96 rows 1.12 / 1.05, 255 rows 1.39 /
// 1.14, 16,320 rows 18.4 / 11.0; 3B shape, 32 rows 0.91 / 1.00, 48 rows 1.04 / 1.02, 64 rows 1.08 / 1.04, 16,320
// rows 30.9 / 17.4; 8 chunks (2 layers, d 128), 1 row 0.27 / 0.23, 16,320 rows 0.57 / 0.29.
constexpr int kPrefillFewRows = 48, kPrefillFewChunks = 16;
constexpr int kBigThreads = 320;
constexpr int kBigRows = 128, kBigCols = 256, kBigStages = 3;
constexpr int kBigStage = kBigCols * 128 + 2 * kBigRows * 128;  // 64 KB
constexpr size_t kBigSmemBytes = 1024 + (size_t)kBigStages * kBigStage;
constexpr size_t kBigPartFloats = (size_t)kBigRows * kBigCols;  // one partial tile

struct BigSmem {
    uint64_t full[kBigStages], empty[kBigStages], acc_full[2], acc_empty[2], drain;
    uint32_t tmem_base;
    int abort, skip, last;
};

// Partial tile of CTA c: slot 2 c + 1 for the tile that it is the first contributor of, else 2 c.
template <int EPI>
__global__ void __launch_bounds__(kBigThreads, 1)
prefill_gemm_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmXlo, GemmParams p,
                    int nout, float *part) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ BigSmem S;
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cta = blockIdx.x;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kBigStages; ++s) { mbar_init(&S.full[s], 1); mbar_init(&S.empty[s], 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(&S.acc_full[a], 1); mbar_init(&S.acc_empty[a], 8); }
        mbar_init(&S.drain, 1);
        S.abort = 0;
        S.skip = *(volatile int *)p.err != 0;  // an earlier kernel of the step reported an error: do nothing
        fence_mbar_init();
        prefetch_tensormap(&tmX);
        prefetch_tensormap(&tmXlo);
    }
    if (warp == 1) { tmem_alloc(&S.tmem_base, 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_base;
    pdl_allow_dependents();
    // (the row count is written before the first kernel of the prefill starts)
    const int rows = S.skip ? 0 : min(*p.rows_dev, p.rows_cap);
    const int nt = (nout + kBigCols - 1) / kBigCols, kch = p.k_chunks;
    const int64_t U = (int64_t)nt * ((rows + kBigRows - 1) / kBigRows) * kch;
    // At most one CTA per unit, so that every CTA between a tile's first and last contributes; with
    // few tiles fewer, so that the time of a CTA's units (~0.5 us each) and of summing a tile's
    // contributors (~1.4 us each) balance, but half of the grid at least: the tensor core's accumulation
    // truncates along a chain, about 1e-9 of the result per element of K, and a CTA's units of a tile are one;
    // half of the grid makes it as long as an even split of 128 x 128 tiles over all of it does.  Relative
    // error against 64 bits and time, with and without that: 80 x 2,048 x 2,048 4.9e-7, 38.7 us / 1.19e-6,
    // 32.9; 255 x 1,536 x 1,536 5.2e-7, 48.3 / 1.10e-6, 41.4; from 300 rows on it changes nothing.
    const int tiles = nt * ((rows + kBigRows - 1) / kBigRows);
    const int G = (int)min64(min64(gridDim.x, U > 0 ? U : 1),
                             max(max(tiles, (int)(gridDim.x + 1) / 2), (int)sqrtf(0.37f * (float)U * (float)tiles) + 1));
    const int64_t u0 = cta < G ? unit_begin(cta, U, G) : 0, u1 = cta < G ? unit_begin(cta + 1, U, G) : 0;
    volatile int *ab = &S.abort;

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        const uint64_t pol_w = l2_policy_evict_last(), pol_x = l2_policy_evict_last();
        int tile = (int)(u0 / kch), kc = (int)(u0 - (int64_t)tile * kch);
        const int n_units = (int)(u1 - u0), n_pre = min(n_units, kBigStages);
        auto load_w = [&](int s, int t, int c) {  // weights of tile t, chunk c; returns nothing: the bytes are expected here
            const int n0 = (t % nt) * kBigCols, n = min(kBigCols, nout - n0);
            bulk_load(ring + s * kBigStage, p.w_blk + ((int64_t)c * nout + n0) * 128, (uint32_t)n * 128, &S.full[s], pol_w);
        };
        // the first stages' weights do not wait for the preceding kernel
        {
            int t = tile, c = kc;
            for (int i = 0; i < n_pre; ++i) {
                if (elect_one()) {
                    mbar_expect_tx(&S.full[i], (uint32_t)min(kBigCols, nout - (t % nt) * kBigCols) * 128);
                    load_w(i, t, c);
                }
                if (++c == kch) { c = 0; ++t; }
            }
        }
        pdl_wait_prior_grids();
        int s = 0, i = 0;
        uint32_t ph = 1;
        bool ok = true;
#pragma unroll 1
        for (; i < n_units; ++i) {
            if (i >= kBigStages) ok = __all_sync(0xffffffffu, mbar_wait(&S.empty[s], ph, p.err) && !*ab);
            if (!ok) break;
            if (elect_one()) {
                uint8_t *x = ring + s * kBigStage + kBigCols * 128;
                const int r0 = tile / nt * kBigRows, n = min(kBigCols, nout - tile % nt * kBigCols);
                mbar_arrive_expect_tx(&S.full[s], (uint32_t)(2 * kBigRows * 128 + (i >= n_pre ? n * 128 : 0)));
                if (i >= n_pre) load_w(s, tile, kc);
                tma_load_2d(x, &tmX, &S.full[s], kc * 64, r0, pol_x);
                tma_load_2d(x + kBigRows * 128, &tmXlo, &S.full[s], kc * 64, r0, pol_x);
            }
            __syncwarp();
            if (++kc == kch) { kc = 0; ++tile; }
            if (++s == kBigStages) { s = 0; ph ^= 1; }
        }
        if (!ok) {  // every load already issued lands before the CTA exits
            *ab = 1;
            for (int q = 0; q < kBigStages && q < i; ++q) {
                const int last = (i - 1 - q) / kBigStages * kBigStages + q;
                mbar_wait(&S.full[q], (uint32_t)((last / kBigStages) & 1), p.err);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        int tile = (int)(u0 / kch), kc = (int)(u0 - (int64_t)tile * kch);
        int s = 0, it = 0;
        uint32_t ph = 0;
        bool ok = true;
#pragma unroll 1
        for (int64_t u = u0; u < u1 && ok; ++it, ++tile, kc = 0) {
            const int a = it & 1;
            if (it >= 2) ok = __all_sync(0xffffffffu, mbar_wait(&S.acc_empty[a], (uint32_t)(((it >> 1) - 1) & 1), p.err));
            tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(a * kBigCols);
            const uint32_t idesc = idesc_bf16_f32(kBigRows, (uint32_t)min(kBigCols, nout - tile % nt * kBigCols));
            const int kc_end = (int)min64(kch, kc + (u1 - u)), kc_first = kc;
            u += kc_end - kc;
#pragma unroll 1
            for (; kc < kc_end && ok; ++kc) {
                ok = __all_sync(0xffffffffu, mbar_wait(&S.full[s], ph, p.err) && !*ab);
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t w = smem_u32(ring) + (uint32_t)(s * kBigStage), x = w + kBigCols * 128;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const uint64_t bd = sdesc_kmajor_sw128(w + kk * 32);
                        tc_mma_bf16(d, sdesc_kmajor_sw128(x + kk * 32), bd, idesc, (kc == kc_first && kk == 0) ? 0u : 1u);
                        tc_mma_bf16(d, sdesc_kmajor_sw128(x + kBigRows * 128 + kk * 32), bd, idesc, 1u);
                    }
                    tc_commit(&S.empty[s]);
                    if (kc + 1 == kc_end) tc_commit(&S.acc_full[a]);
                }
                __syncwarp();
                if (++s == kBigStages) { s = 0; ph ^= 1; }
            }
        }
        if (!ok) *ab = 1;
        if (elect_one()) tc_commit(&S.drain);
        mbar_wait(&S.drain, 0, p.err);  // every MMA has retired before tensor memory is released
    } else {
        // ------------------------------------------------------------ epilogue
        pdl_wait_prior_grids();
        const int quarter = warp & 3, half = (warp - 2) >> 2, lrow = quarter * 32 + lane, etid = threadIdx.x - 64;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        int tile = (int)(u0 / kch), kc = (int)(u0 - (int64_t)tile * kch), it = 0;
#pragma unroll 1
        for (int64_t u = u0; u < u1; ++it, ++tile, kc = 0) {
            const int a = it & 1;
            const int kc_end = (int)min64(kch, kc + (u1 - u));
            const bool whole = kc == 0 && kc_end == kch;
            u += kc_end - kc;
            const int r = tile / nt * kBigRows + lrow, n0 = tile % nt * kBigCols + half * 128;
            const bool live = r < rows, cols = n0 < nout && r - lane < rows;  // (a warp of 32 rows past the end: nothing)
            // the row's scale and place, read while the MMAs run
            float rs = 0.f;
            int pos = 0, slot = 0;
            if ((EPI == EPI_QKV || EPI == EPI_SWIGLU) && live) {
                float ss = 0.f;
#pragma unroll 4
                for (int t = 0; t < p.ssq_tiles; ++t) ss += __ldcg(&p.ssq[(int64_t)t * p.rows_cap + r]);
                rs = rsqrtf(ss * p.inv_dim + p.eps);
                if (EPI == EPI_QKV) { pos = p.row_pos[r]; slot = p.row_slot[r]; }
            }
            if (!mbar_wait(&S.acc_full[a], (uint32_t)((it >> 1) & 1), p.err)) *ab = 1;
            tc_fence_after();
            // (one decision for all eight warps: none is left in a barrier)
            named_bar_sync(1, 256);
            const bool stop = *ab != 0;
            named_bar_sync(1, 256);
            if (stop) break;
            int ca = cta, cb = cta;
            bool finish = whole;
            if (!whole) {
                ca = cta_of_unit((int64_t)tile * kch, U, G);
                cb = cta_of_unit((int64_t)(tile + 1) * kch - 1, U, G);
                float *mine = part + (size_t)(2 * cta + (cta == ca ? 1 : 0)) * kBigPartFloats + half * 128 * kBigRows + lrow;
                if (cols) {
#pragma unroll 1
                    for (int cc = 0; cc < 4; ++cc) {
                        float v[32];
                        tmem_ld_32x32b_x32(tmem + lane_base + (uint32_t)(a * kBigCols + half * 128 + cc * 32), v);
#pragma unroll
                        for (int e = 0; e < 32; ++e) mine[(cc * 32 + e) * kBigRows] = v[e];
                    }
                }
                __threadfence();
                named_bar_sync(1, 256);
                if (etid == 0) {
                    const int old = atom_add_acq_rel_gpu(&p.ws_cnt[tile], 1);
                    S.last = old == cb - ca;
                    if (S.last) p.ws_cnt[tile] = 0;
                }
                named_bar_sync(1, 256);
                finish = S.last != 0;
                __threadfence();
            }
            float sq = 0.f;
            if (finish && cols) {
#pragma unroll 1
                for (int cc = 0; cc < 4; ++cc) {
                    float v[32];
                    if (whole) {
                        tmem_ld_32x32b_x32(tmem + lane_base + (uint32_t)(a * kBigCols + half * 128 + cc * 32), v);
                    } else {
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[e] = 0.f;
#pragma unroll 1
                        for (int c = ca; c <= cb; c += 2) {  // in CTA order, two contributors' loads in flight
                            const int off = (half * 128 + cc * 32) * kBigRows + lrow;
                            const float *s0 = part + (size_t)(2 * c + (c == ca ? 1 : 0)) * kBigPartFloats + off;
                            const float *s1 = part + (size_t)(2 * c + 2) * kBigPartFloats + off;
                            float w0[32], w1[32];
#pragma unroll
                            for (int e = 0; e < 32; ++e) w0[e] = __ldcg(s0 + e * kBigRows);
#pragma unroll
                            for (int e = 0; e < 32; ++e) w1[e] = c < cb ? __ldcg(s1 + e * kBigRows) : 0.f;
#pragma unroll
                            for (int e = 0; e < 32; ++e) v[e] = (v[e] + w0[e]) + w1[e];
                        }
                    }
                    if (!live) continue;
                    const int n = n0 + cc * 32;
                    if constexpr (EPI == EPI_QKV) {
                        // units of 16: 8 dims of a head's first half and their rotation partners
                        const int hd = p.head_dim, half_hd = hd >> 1;
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            const int nu = n + 16 * q, head = nu / hd, fi = (nu - head * hd) / 2;
                            float lo[8], hi[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) { lo[e] = v[16 * q + e] * rs; hi[e] = v[16 * q + 8 + e] * rs; }
                            if (head < p.n_heads + p.n_kv) {
                                const float4 *cs = reinterpret_cast<const float4 *>(p.rope + (int64_t)pos * half_hd + fi);
#pragma unroll
                                for (int e = 0; e < 8; e += 2) {
                                    const float4 c = __ldg(cs + e / 2);
                                    const float x0 = lo[e], y0 = hi[e], x1 = lo[e + 1], y1 = hi[e + 1];
                                    lo[e] = x0 * c.x - y0 * c.y;
                                    hi[e] = y0 * c.x + x0 * c.y;
                                    lo[e + 1] = x1 * c.z - y1 * c.w;
                                    hi[e + 1] = y1 * c.z + x1 * c.w;
                                }
                            }
                            uint16_t *dst;
                            if (head < p.n_heads) {
                                dst = p.q_out + (int64_t)r * (p.n_heads * hd) + head * hd + fi;
                            } else {
                                const int isv = head >= p.n_heads + p.n_kv, kvh = head - p.n_heads - isv * p.n_kv;
                                dst = p.kv + (int64_t)slot * p.kv_slot_stride +
                                      ((int64_t)(isv * p.n_kv + kvh) * p.kv_cap + pos) * hd + fi;
                            }
                            uint16_t h[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) h[e] = f32_to_f16_sat(lo[e]);
                            *reinterpret_cast<uint4 *>(dst) = pack8(h);
#pragma unroll
                            for (int e = 0; e < 8; ++e) h[e] = f32_to_f16_sat(hi[e]);
                            *reinterpret_cast<uint4 *>(dst + half_hd) = pack8(h);
                        }
                    } else if constexpr (EPI == EPI_SWIGLU) {
#pragma unroll
                        for (int q = 0; q < 2; ++q) {  // 8 gate, 8 up
                            uint16_t h[8], l[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                const float gv = v[16 * q + e] * rs, uv = v[16 * q + 8 + e] * rs;
                                split_bf16(gv / (1.0f + expf(-gv)) * uv, h[e], l[e]);
                            }
                            const int64_t idx = (int64_t)r * p.ld + (n + 16 * q) / 2;
                            *reinterpret_cast<uint4 *>(p.h_out + idx) = pack8(h);
                            *reinterpret_cast<uint4 *>(p.h_lo + idx) = pack8(l);
                        }
                    } else {
                        const int64_t idx = (int64_t)r * p.ld + n;
                        float4 x[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) x[e] = __ldcg(reinterpret_cast<const float4 *>(p.x_f32 + idx) + e);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const uint4 gb = __ldg(reinterpret_cast<const uint4 *>(p.g_next + n) + q);
                            const uint32_t gw[4] = {gb.x, gb.y, gb.z, gb.w};
                            uint16_t h[8], l[8];
                            float y[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                const float4 xv = x[2 * q + (e >> 2)];
                                const float xo = (e & 3) == 0 ? xv.x : (e & 3) == 1 ? xv.y : (e & 3) == 2 ? xv.z : xv.w;
                                y[e] = xo + v[8 * q + e];
                                sq += y[e] * y[e];
                                split_bf16(y[e] * bf16_to_f32((uint16_t)(gw[e >> 1] >> (16 * (e & 1)))), h[e], l[e]);
                            }
                            float4 *xd = reinterpret_cast<float4 *>(p.x_f32 + idx) + 2 * q;
                            xd[0] = make_float4(y[0], y[1], y[2], y[3]);
                            xd[1] = make_float4(y[4], y[5], y[6], y[7]);
                            *(reinterpret_cast<uint4 *>(p.xg_out + idx) + q) = pack8(h);
                            *(reinterpret_cast<uint4 *>(p.xg_lo + idx) + q) = pack8(l);
                        }
                    }
                }
                if (EPI == EPI_RESID && live) p.ssq_out[(int64_t)(n0 / 128) * p.rows_cap + r] = sq;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.acc_empty[a]);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, 512);
}

}  // namespace sara
