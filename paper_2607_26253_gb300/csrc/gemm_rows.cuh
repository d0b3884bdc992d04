// The projection GEMM of up to 128 activation rows as a call of its own:
//     Y[r][n] = sum_c X[r][c] * W[n][c]        (bf16 in, fp32 accumulation and result)
// bound by reading W.  The weight tile is the MMA's A operand (M = 128 output features), the
// activation rows are B (N = rows rounded up to 16), the accumulator lives in tensor memory.
// Operands come by TMA (128-byte swizzle) through an mbarrier ring of about 100 KB a CTA, two
// CTAs an SM, so that ~190 KB of loads are in flight per SM.
//
// Work split: with at least two tiles of 128 features per SM, CTAs walk whole tiles (two
// accumulators, so a tile's epilogue overlaps the next tile's MMAs).  With fewer, a cluster of
// 2, 4 or 8 CTAs shares a tile, each a contiguous share of K; their partial tiles meet in
// distributed shared memory, where each CTA sums its share of the rows in rank order: no
// workspace, no atomics, the same sums on every run.  Against a stream-K split over all SMs folded
// by 64-bit fixed-point atomics (with four 16 KB weight stages in flight an SM), whole calls:
// 1 x 2,048 x 1,536: 18.4 -> 12.4 us; 64 x 151,936 x 1,536: 122 -> 81 us (6.2 TB/s); through the
// allocation-free entry point (which also cleared 8 MiB a call) 33 x 2,048 x 11,008: 45 -> 15 us.
//
// Warp roles (192 threads): warp 0 TMA producer, warp 1 MMA issuer and tensor-memory owner,
// warps 2..5 epilogue (warp w reads tensor-memory lanes 32 (w % 4) ..).
#pragma once
#include "device_common.cuh"
#include "host_util.h"

namespace sara {

constexpr int kRowsThreads = 192;
constexpr int kRowsTileM = 128;   // features per tile
constexpr int kRowsTileK = 64;    // reduction elements per stage (128 B of bf16)
constexpr int kRowsMax = 128;     // activation rows
constexpr int kRowsBox = 32;      // activation rows per TMA box
constexpr int kRowsMaxStages = 5;
constexpr int kRowsRing = 104 * 1024;  // ring bytes at most: two CTAs fit an SM
constexpr int kRowsMaxSplit = 8;

struct GemmRowsParams {
    int tiles, kch, R, nout, split, stages;
    float *y;  // [R][nout]
};
struct GemmRowsSmem {
    uint64_t full[kRowsMaxStages], empty[kRowsMaxStages], acc_full[2], acc_empty[2], drain;
    uint32_t tmem_base;
    int abort;
};
__host__ __device__ inline int gemm_rows_stage(int R) {
    return kRowsTileM * 128 + (R + kRowsBox - 1) / kRowsBox * kRowsBox * 128;
}

static __global__ void __launch_bounds__(kRowsThreads)
gemm_rows_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, GemmRowsParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ GemmRowsSmem S;
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) { mbar_init(&S.full[s], 1); mbar_init(&S.empty[s], 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(&S.acc_full[a], 1); mbar_init(&S.acc_empty[a], 4); }
        mbar_init(&S.drain, 1);
        S.abort = 0;
        fence_mbar_init();
        prefetch_tensormap(&tmW);
        prefetch_tensormap(&tmX);
    }
    if (warp == 1) { tmem_alloc(&S.tmem_base, 256); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_base;
    const int rank = (int)blockIdx.x % p.split, unit = (int)blockIdx.x / p.split, units = (int)gridDim.x / p.split;
    const int kc0 = rank * p.kch / p.split, kc1 = (rank + 1) * p.kch / p.split;
    const int nbox = (p.R + kRowsBox - 1) / kRowsBox;
    const int stage = gemm_rows_stage(p.R);
    volatile int *ab = &S.abort;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        const uint64_t pol_w = l2_policy_evict_first(), pol_x = l2_policy_evict_last();
        int s = 0, issued = 0;
        uint32_t ph = 1;
        bool ok = true;
#pragma unroll 1
        for (int t = unit; t < p.tiles && ok; t += units)
#pragma unroll 1
            for (int kc = kc0; kc < kc1; ++kc, ++issued) {
                if (issued >= p.stages) ok = __all_sync(0xffffffffu, mbar_wait(&S.empty[s], ph, nullptr)) && !*ab;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                uint8_t *w = ring + s * stage;
                if (elect_one()) {
                    mbar_arrive_expect_tx(&S.full[s], (uint32_t)stage);
                    tma_load_2d(w, &tmW, &S.full[s], kc * kRowsTileK, t * kRowsTileM, pol_w);
#pragma unroll 1
                    for (int b = 0; b < nbox; ++b)
                        tma_load_2d(w + kRowsTileM * 128 + b * kRowsBox * 128, &tmX, &S.full[s], kc * kRowsTileK, b * kRowsBox,
                                    pol_x);
                }
                if (++s == p.stages) { s = 0; ph ^= 1; }
            }
        if (!ok) {  // every load already issued lands before the CTA exits
            *ab = 1;
            for (int q = 0; q < p.stages && q < issued; ++q) {
                const int last = (issued - 1 - q) / p.stages * p.stages + q;
                mbar_wait(&S.full[q], (uint32_t)((last / p.stages) & 1), nullptr);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        const uint32_t idesc = idesc_bf16_f32(128, (uint32_t)((p.R + 15) & ~15));
        int s = 0, it = 0;
        uint32_t ph = 0;
        bool ok = true;
#pragma unroll 1
        for (int t = unit; t < p.tiles && ok; t += units, ++it) {
            const int a = it & 1;
            if (it >= 2) ok = __all_sync(0xffffffffu, mbar_wait(&S.acc_empty[a], (uint32_t)(((it >> 1) - 1) & 1), nullptr));
            tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(a * 128);
#pragma unroll 1
            for (int kc = kc0; kc < kc1 && ok; ++kc) {
                ok = __all_sync(0xffffffffu, mbar_wait(&S.full[s], ph, nullptr) && !*ab);
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t aw = smem_u32(ring) + (uint32_t)(s * stage), ax = aw + kRowsTileM * 128;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        tc_mma_bf16(d, sdesc_kmajor_sw128(aw + kk * 32), sdesc_kmajor_sw128(ax + kk * 32), idesc,
                                    (kc == kc0 && kk == 0) ? 0u : 1u);
                    tc_commit(&S.empty[s]);
                    if (kc + 1 == kc1) tc_commit(&S.acc_full[a]);
                }
                __syncwarp();
                if (++s == p.stages) { s = 0; ph ^= 1; }
            }
        }
        if (!ok) *ab = 1;
        if (elect_one()) tc_commit(&S.drain);
        mbar_wait(&S.drain, 0, nullptr);  // every MMA has retired before tensor memory is released
    } else {
        // ------------------------------------------------------------ epilogue
        const int quarter = warp & 3, mrow = quarter * 32 + lane;
        int it = 0;
#pragma unroll 1
        for (int t = unit; t < p.tiles; t += units, ++it) {
            const int a = it & 1;
            if (!mbar_wait(&S.acc_full[a], (uint32_t)((it >> 1) & 1), nullptr)) *ab = 1;
            if (__any_sync(0xffffffffu, *ab != 0)) break;
            tc_fence_after();
            // feature mrow of the tile, 32 rows at a time: straight to Y, or to this CTA's partial
            // tile in the (now idle) ring
            float *dst = p.split == 1 ? p.y + (int64_t)t * kRowsTileM + mrow : reinterpret_cast<float *>(ring) + mrow;
            const int64_t ld = p.split == 1 ? p.nout : kRowsTileM;
#pragma unroll 1
            for (int c0 = 0; c0 < p.R; c0 += 32) {
                float v[32];
                tmem_ld_32x32b_x32(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(a * 128 + c0), v);
#pragma unroll
                for (int c = 0; c < 32; ++c)
                    if (c0 + c < p.R) dst[(c0 + c) * ld] = v[c];
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.acc_empty[a]);
        }
    }
    __syncwarp();
    if (p.split > 1) {
        // one tile per cluster: the CTAs' partial tiles summed in rank order, rows dealt out
        cluster_sync();
        if (warp >= 2 && unit < p.tiles) {
            const int mrow = (warp & 3) * 32 + lane;
#pragma unroll 1
            for (int r = rank; r < p.R; r += p.split) {
                const float *src = reinterpret_cast<const float *>(ring) + r * kRowsTileM + mrow;
                float v[kRowsMaxSplit];
#pragma unroll
                for (int q = 0; q < kRowsMaxSplit; ++q) v[q] = q < p.split ? ld_cluster_f32(cluster_addr(src, q)) : 0.f;
                // compensated (Knuth's two-sum): splitting K adds no rounding of its own; an infinite
                // or NaN sum has no error term
                float s = v[0], c = 0.f;
#pragma unroll
                for (int q = 1; q < kRowsMaxSplit; ++q) {
                    const float t = __fadd_rn(s, v[q]), b = __fsub_rn(t, s);
                    c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(v[q], b)));
                    s = t;
                }
                p.y[(int64_t)r * p.nout + unit * kRowsTileM + mrow] = isfinite(s) ? __fadd_rn(s, c) : s;
            }
        }
        cluster_sync();  // no CTA leaves while its partial tile is read
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, 256);
}

// Launch for X [R][K], W [nout][K], Y [R][nout]; 1 <= R <= 128, nout % 128 == 0, K % 64 == 0.
// The split doubles until the CTAs fill the SMs twice (two fit an SM), within K and 8.
inline void launch_gemm_rows(cudaStream_t s, int sms, const uint16_t *X, const uint16_t *W, float *Y, int R, int nout, int K) {
    GemmRowsParams p{};
    p.tiles = nout / kRowsTileM;
    p.kch = K / kRowsTileK;
    p.R = R;
    p.nout = nout;
    p.y = Y;
    const int stage = gemm_rows_stage(R);
    p.stages = kRowsRing / stage < kRowsMaxStages ? kRowsRing / stage : kRowsMaxStages;
    p.split = 1;
    while (p.split < kRowsMaxSplit && 2 * p.split <= p.kch && p.tiles * 2 * p.split <= 2 * sms) p.split *= 2;
    const int grid = p.split > 1 ? p.tiles * p.split : (p.tiles < 2 * sms ? p.tiles : 2 * sms);
    const size_t smem = 1024 + (size_t)p.stages * stage;
    const CUtensorMap tw = make_tmap_bf16(W, K, nout, kRowsTileK, kRowsTileM);
    const CUtensorMap tx = make_tmap_bf16(X, K, R, kRowsTileK, kRowsBox);
    launch_cluster(s, false, dim3((unsigned)grid), dim3(kRowsThreads), smem, (unsigned)p.split, gemm_rows_kernel, tw, tx, p);
}

// SM count of the current device, its kernel attributes set (looked up once per device).
int gemm_rows_sms();

}  // namespace sara
