// The projection GEMM of up to 128 activation rows as a call of its own:
//     Y[r][n] = sum_c X[r][c] * W[n][c]        (bf16 in, fp32 accumulation and result)
// bound by reading W.  The weight tile is the MMA's A operand (M = 128 output features), the
// activation rows are B (N = rows rounded up to 16), the accumulator lives in tensor memory.
// Operands come by TMA (128-byte swizzle) through an mbarrier ring of about 100 KB a CTA, two
// CTAs an SM, so that ~190 KB of loads are in flight per SM.
//
// Work split: with at least two tiles of 128 features per SM, CTAs walk whole tiles.  With fewer, a
// cluster of 2, 4 or 8 CTAs shares a tile, each a contiguous share of K; their partial tiles meet in
// distributed shared memory, where each CTA sums its share of the rows: no workspace, no
// atomics, the same sums on every run.
//
// Accuracy: the tensor core's accumulation truncates, which costs about 1e-9 of the result for every
// element of K in one chain (measured at 64 .. 11,008).  So a CTA's share is accumulated in segments of
// `chain` chunks at most, in turn in several tensor-memory buffers, and the epilogue adds them in fp32; where the
// roundings of these sums would show beside so short a chain (few tiles: `carry`), with their errors
// carried along (Knuth's two-sum).  Relative error: 64 x 151,936 x 1,536 7.7e-7, against 1.5e-6 in one chain;
// 8 x 128 x 2,368 6.7e-8 (the rounding of the result and chains of 64), against 2.8e-7.
//
// Kernel times (back to back in a graph): 1 x 2,048 x 1,536 6.0 us, 33 x 2,048 x 11,008 14.2, 64 x 2,048 x 1,536
// 8.7, 64 x 151,936 x 1,536 72.4 (6.4 TB/s), 128 x 17,920 x 1,536 14.3, 128 x 151,936 x 1,536 87.8; in one chain
// per share, with four epilogue warps and two buffers: 5.2, 13.4, 7.6, 71.1, 27.1, 87.2.
//
// Warp roles (320 threads): warp 0 TMA producer, warp 1 MMA issuer and tensor-memory owner, warps 2..9
// epilogue (warp w: tensor-memory lanes 32 (w % 4) .., half (w - 2) / 4 of the rows).
#pragma once
#include "device_common.cuh"
#include "host_util.h"

namespace sara {

constexpr int kRowsTileM = 128;   // features per tile
constexpr int kRowsTileK = 64;    // reduction elements per stage (128 B of bf16)
constexpr int kRowsMax = 128;     // activation rows
constexpr int kRowsBox = 32;      // activation rows per TMA box
constexpr int kRowsMaxStages = 5;
constexpr int kRowsMaxSplit = 8;
constexpr int kRowsThreads = 320;
constexpr int kRowsRing = 104 * 1024;  // ring bytes at most: two CTAs fit an SM
// C: rows of an epilogue thread, 32 or 64 (kernel template); accumulators in a CTA's 256 tensor-memory columns
__host__ __device__ constexpr int rows_bufs(int C) { return 128 / C; }

struct GemmRowsParams {
    int tiles, kch, R, nout, split, stages, chain;
    bool carry;  // the segments' rounding errors are carried along
    float *y;  // [R][nout]
};
struct GemmRowsSmem {
    uint64_t full[kRowsMaxStages], empty[kRowsMaxStages], acc_full[4], acc_empty[4], drain;
    uint32_t tmem_base;
    int abort;
};
__host__ __device__ inline int gemm_rows_stage(int R) {
    return kRowsTileM * 128 + (R + kRowsBox - 1) / kRowsBox * kRowsBox * 128;
}
// s += v, the rounding error and v's own (e) to c.  Below: two sums at once, without e.
__device__ __forceinline__ void two_sum(float &s, float &c, float v, float e) {
    const float t = __fadd_rn(s, v), b = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(v, b))));
    s = t;
}
__device__ __forceinline__ void two_sum(uint64_t &s, uint64_t &c, uint64_t v) {
    const uint64_t t = add_f32x2(s, v), b = sub_f32x2(t, s);
    c = add_f32x2(c, add_f32x2(sub_f32x2(s, sub_f32x2(t, b)), sub_f32x2(v, b)));
    s = t;
}
// The sum; an infinite or NaN one has no error term.
__device__ __forceinline__ float sum_of(float s, float c) { return isfinite(s) ? __fadd_rn(s, c) : s; }

template <int C>
__global__ void __launch_bounds__(kRowsThreads, 2)
gemm_rows_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, GemmRowsParams p) {
    constexpr int kBufs = rows_bufs(C);
    extern __shared__ uint8_t smem_raw[];
    __shared__ GemmRowsSmem S;
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) { mbar_init(&S.full[s], 1); mbar_init(&S.empty[s], 1); }
        for (int a = 0; a < kBufs; ++a) { mbar_init(&S.acc_full[a], 1); mbar_init(&S.acc_empty[a], 8); }
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
    const int row0 = (int)blockIdx.y * 2 * C, R = min(2 * C, p.R - row0);  // this CTA's rows
    const int rank = (int)blockIdx.x % p.split, unit = (int)blockIdx.x / p.split, units = (int)gridDim.x / p.split;
    const int kc0 = rank * p.kch / p.split, kc1 = (rank + 1) * p.kch / p.split;
    const int nseg = (kc1 - kc0 + p.chain - 1) / p.chain;
    auto seg_end = [&](int i) { return kc0 + (i + 1) * (kc1 - kc0) / nseg; };  // chunks of segment i: up to here
    const int nbox = (R + kRowsBox - 1) / kRowsBox;
    const int stage = gemm_rows_stage(R);
    const bool carry = C == 32 && p.carry;
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
                        tma_load_2d(w + kRowsTileM * 128 + b * kRowsBox * 128, &tmX, &S.full[s], kc * kRowsTileK, row0 + b * kRowsBox,
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
        const uint32_t idesc = idesc_bf16_f32(128, (uint32_t)((R + 15) & ~15));
        int s = 0, it = 0;
        uint32_t ph = 0;
        bool ok = true;
#pragma unroll 1
        for (int t = unit; t < p.tiles && ok; t += units) {
            int kc = kc0;
#pragma unroll 1
            for (int i = 0; i < nseg && ok; ++i, ++it) {
                const int a = it % kBufs, first = kc, end = seg_end(i);
                if (it >= kBufs)
                    ok = __all_sync(0xffffffffu, mbar_wait(&S.acc_empty[a], (uint32_t)((it / kBufs - 1) & 1), nullptr));
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(a * 2 * C);
#pragma unroll 1
                for (; kc < end && ok; ++kc) {
                    ok = __all_sync(0xffffffffu, mbar_wait(&S.full[s], ph, nullptr) && !*ab);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        const uint32_t aw = smem_u32(ring) + (uint32_t)(s * stage), ax = aw + kRowsTileM * 128;
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            tc_mma_bf16(d, sdesc_kmajor_sw128(aw + kk * 32), sdesc_kmajor_sw128(ax + kk * 32), idesc,
                                        (kc == first && kk == 0) ? 0u : 1u);
                        tc_commit(&S.empty[s]);
                        if (kc + 1 == end) tc_commit(&S.acc_full[a]);
                    }
                    __syncwarp();
                    if (++s == p.stages) { s = 0; ph ^= 1; }
                }
            }
        }
        if (!ok) *ab = 1;
        if (elect_one()) tc_commit(&S.drain);
        mbar_wait(&S.drain, 0, nullptr);  // every MMA has retired before tensor memory is released
    } else {
        // ------------------------------------------------------------ epilogue
        // this thread: feature mrow of the tile, rows r0 .. r0 + C - 1; sums and their rounding errors
        const int quarter = warp & 3, mrow = quarter * 32 + lane, r0 = (warp - 2) / 4 * C;
        uint64_t sum[C / 2], err[C == 32 ? C / 2 : 1];  // (two rows each)
        int it = 0;
        bool ok = true;
#pragma unroll 1
        for (int t = unit; t < p.tiles && ok; t += units) {
#pragma unroll
            for (int c = 0; c < C / 2; ++c) {
                sum[c] = 0;
                if (C == 32) err[c] = 0;
            }
#pragma unroll 1
            for (int i = 0; i < nseg; ++i, ++it) {
                const int a = it % kBufs;
                if (!mbar_wait(&S.acc_full[a], (uint32_t)((it / kBufs) & 1), nullptr)) *ab = 1;
                ok = !__any_sync(0xffffffffu, *ab != 0);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int c0 = 0; c0 < C; c0 += 16)
                    if (r0 + c0 < R) {
                        uint64_t v[8];
                        tmem_ld_32x32b_x16(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(a * 2 * C + r0 + c0), v);
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            if (carry) two_sum(sum[c0 / 2 + c], err[C == 32 ? c0 / 2 + c : 0], v[c]);
                            else sum[c0 / 2 + c] = add_f32x2(sum[c0 / 2 + c], v[c]);
                        }
                    }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.acc_empty[a]);
            }
            if (!ok) break;
            // straight to Y, or sums and errors to this CTA's part of the (now idle) ring: [2][R][128]
            const bool whole = p.split == 1;
            float *dst = whole ? p.y + (int64_t)(row0 + r0) * p.nout + t * kRowsTileM + mrow
                               : reinterpret_cast<float *>(ring) + r0 * kRowsTileM + mrow;
            const int64_t ld = whole ? p.nout : kRowsTileM, lo = R * kRowsTileM;
#pragma unroll
            for (int c = 0; c < C; ++c, dst += ld) {
                if (r0 + c >= R) break;
                const float x = __uint_as_float((uint32_t)(sum[c / 2] >> (32 * (c & 1))));
                const float e = carry ? __uint_as_float((uint32_t)(err[C == 32 ? c / 2 : 0] >> (32 * (c & 1)))) : 0.f;
                dst[0] = whole ? sum_of(x, e) : x;
                if (!whole && carry) dst[lo] = e;
            }
        }
    }
    __syncwarp();
    if (p.split > 1) {
        // one tile per cluster: the CTAs' partial tiles summed from this CTA's own on (each CTA reading another's at
        // a time: in rank order they would all queue up at the same one), rows dealt out
        cluster_sync();
        if (warp >= 2 && unit < p.tiles) {
            const int mrow = (warp & 3) * 32 + lane;
#pragma unroll 1
            for (int r = rank + (warp - 2) / 4 * p.split; r < R; r += 2 * p.split) {
                const float *src = reinterpret_cast<const float *>(ring) + r * kRowsTileM + mrow;
                float v[kRowsMaxSplit], e[kRowsMaxSplit];
#pragma unroll
                for (int q = 0; q < kRowsMaxSplit; ++q) {
                    const uint32_t from = (uint32_t)((rank + q) & (p.split - 1));
                    v[q] = q < p.split ? ld_cluster_f32(cluster_addr(src, from)) : 0.f;
                    e[q] = q < p.split && carry ? ld_cluster_f32(cluster_addr(src + R * kRowsTileM, from)) : 0.f;
                }
                float s = v[0], c = e[0];
#pragma unroll
                for (int q = 1; q < kRowsMaxSplit; ++q) two_sum(s, c, v[q], e[q]);
                p.y[(int64_t)(row0 + r) * p.nout + unit * kRowsTileM + mrow] = sum_of(s, c);
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
// More than 64 rows: in two halves, which read W twice (mostly from L2), up to a tile per SM; above, whole (128 x
// 2,048 x 11,008: 16.2 us against 18.8 whole; 128 x 151,936 x 1,536: 97 against 89).  The split doubles until
// the CTAs fill the SMs twice, within K and 8.
template <int C>
inline void launch_gemm_rows_c(cudaStream_t s, int sms, const uint16_t *X, const uint16_t *W, float *Y, int R, int nout, int K) {
    GemmRowsParams p{};
    p.tiles = nout / kRowsTileM;
    p.kch = K / kRowsTileK;
    p.R = R;
    p.nout = nout;
    p.y = Y;
    const int parts = (R + 2 * C - 1) / (2 * C);
    const int stage = gemm_rows_stage(R < 2 * C ? R : 2 * C), slots = 2 * sms / parts;
    p.stages = kRowsRing / stage < kRowsMaxStages ? kRowsRing / stage : kRowsMaxStages;
    p.split = 1;
    while (C == 32 && p.split < kRowsMaxSplit && 2 * p.split <= p.kch && (int64_t)p.tiles * 2 * p.split <= slots) p.split *= 2;
    // A chain of at most half of the chunks that an even split over the SMs gives one (a single chunk at least).  Errors
    // are carried where that is no more than 64 .. 112 elements, or sums are of more than 8 segments: each plain
    // sum rounds by 2.4e-8 of its value (root mean square), a chain of 64 by 6.4e-8 of the result.
    const int64_t even = (int64_t)p.tiles * p.kch / sms;
    p.chain = (int)(even < p.kch ? even : p.kch) / 2;
    if (p.chain < 1) p.chain = 1;
    const int nseg = ((p.kch + p.split - 1) / p.split + p.chain - 1) / p.chain;
    p.carry = 4 * (int64_t)p.tiles * p.kch < 7 * sms || nseg > 8;
    const int grid = p.split > 1 ? p.tiles * p.split : (p.tiles < slots ? p.tiles : slots);
    const size_t smem = 1024 + (size_t)p.stages * stage;
    const CUtensorMap tw = make_tmap_bf16(W, K, nout, kRowsTileK, kRowsTileM);
    const CUtensorMap tx = make_tmap_bf16(X, K, R, kRowsTileK, kRowsBox);
    launch_cluster(s, false, dim3((unsigned)grid, (unsigned)parts), dim3(kRowsThreads), smem, (unsigned)p.split,
                   gemm_rows_kernel<C>, tw, tx, p);
}
inline void launch_gemm_rows(cudaStream_t s, int sms, const uint16_t *X, const uint16_t *W, float *Y, int R, int nout, int K) {
    if (R <= 64 || nout / kRowsTileM <= sms) launch_gemm_rows_c<32>(s, sms, X, W, Y, R, nout, K);
    else launch_gemm_rows_c<64>(s, sms, X, W, Y, R, nout, K);
}

// SM count of the current device, its kernel attributes set (looked up once per device).
int gemm_rows_sms();

}  // namespace sara
