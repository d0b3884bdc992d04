// One decode step of the policy (embedding -> every layer -> lm_head logits) as a single
// persistent, cooperative kernel: one CTA per SM, phases separated
// by release/acquire arrival counters in global memory instead of kernel boundaries.
//
// Why: at decode batch sizes the per-layer work is a few MB of weights per projection, so
// a kernel per projection spends most of its time starting, filling its pipeline and
// draining.  Here the weight stream never stops: the producer warp walks the whole step's
// weight tiles (and the attention phase's KV blocks, which do not depend on this step's
// activations) ahead of the consumers through a ring of 32 KB shared-memory slots, across
// phase boundaries.  Only the small activation operands wait for the previous phase.
//
// GEMM orientation: the activation rows are the MMA's M and 256 weight rows its N, so one
// tcgen05.mma (K = 16) consumes 8 KB of weights (~133 cycles at M = 64 or 128 alike).  The
// activation is a bf16 hi/lo pair (~16 mantissa bits); up to 64 live rows both parts sit in
// one stacked operand and a k-step is one MMA, above that two MMAs (hi, lo) accumulate.
// Rows beyond the live count are don't-care.
//
// Split-K: a phase's (tile, k-chunk) units are cut into equal contiguous ranges over its
// CTAs; each CTA stores its fp32 partial tile with plain stores and the consuming phase
// sums a tile's partials in CTA order (deterministic, no atomics).  Gate / up, lm_head and, up to
// 8 rows, q/k/v and O are column-owned instead: each CTA takes 16-feature units with the whole K
// and applies what follows in its epilogue (no partials, no finalisation phase).
//
// Warp roles (352 threads, 11 warps):
//   warp 0   W producer: bulk copies of pre-swizzled weight tiles and KV blocks
//   warp 1   tcgen05 issuer and tensor-memory owner; hands the attention phase's KV tiles
//            to the compute warp group that runs their unit
//   warp 2   X producer: activation chunks, after the phase they come from has completed
//   warps 3..10  compute: GEMM epilogues, attention, residual + RMSNorm finalisation, embedding,
//                logits
//
// Phases of layer l (counter index 1 + 9l + k):
//   0 QKV   x_g W_qkv^T -> partials        (a subset of the CTAs: few tiles)
//   2 ATT   q, k, v = RMSNorm scale + RoPE of the summed partials, fp16 (counter 1: of the few rows'
//           q/k/v phase, which does that itself); softmax(q K^T) V, 128-position KV blocks,
//           online softmax over a split's blocks with warp-level MMAs (mma.sync: N = 8 heads,
//           operands and accumulators in registers, no exchange between warps inside a split; the
//           tcgen05 path's issue / commit / tensor-memory round trips cost more than these
//           products); the new k, v join the tiles and the KV cache here; the last split of a row
//           to finish merges the splits
//   3 O     att W_o^T -> partials           (a subset of the CTAs)
//   4 FIN_O x += sum; x_g = x * g_mlp (bf16 hi/lo, blocked); per-row sum of squares
//   6 GU    h = silu(r g) * (r u), g | u = x_g W_gu^T, r = 1/rms(x)  (bf16 hi/lo, blocked): gate
//           and up rows alternate in blocks of 8, a CTA holds whole features (counter 5 is unused)
//   7 DOWN  h W_down^T -> partials
//   8 FIN_D x += sum; x_g = x * g_next; sum of squares
// then lm_head, column-owned and fused with the Gumbel-max sampler: per (row, CTA, half of its columns)
// maximum of logit + noise; the logits are stored only under teacher forcing.
//
// Layouts (all chosen so that bulk copies land MMA operands in shared memory in the
// 128-byte-swizzled K-major form the tensor core reads):
//   weights       chunk-major [K/64][N][64], 16-byte granule j of row r at granule j ^ (r % 8):
//                 any 8-aligned run of rows of a chunk is one contiguous copy
//   activations   [K/64][2 rows16][64] bf16, 8-row groups alternating hi / lo parts, same swizzle
//   KV cache      per (layer, slot, kv head, 128-position block): K as [d/64][128 pos][64 d]
//                 and V transposed as [pos/64][128 d][64 pos], fp16, head dim padded to 128
#pragma once
#include "device_common.cuh"
#include "step_state.cuh"

namespace sara {

constexpr int kMegaThreads = 352;
constexpr int kMegaCThreads = 256;  // compute warps 3..10
constexpr int kMaxWSlots = 5;  // weight / KV ring entries of a launch: ring_slots
constexpr int kSlotBytes = 32768;
constexpr int kRingBytes = 5 * kSlotBytes + 53248;  // W slots, then the X stages
constexpr int kMaxXStages = 8;
constexpr int kTileN = 256;           // weight rows (output features) per GEMM tile
constexpr int kKVPos = 128;           // positions per KV block (an attention split holds `span` blocks)
constexpr int kKVBlockBytes = 65536;  // K 2 x 16 KB + V^T 2 x 16 KB
constexpr int kMegaMaxSplits = 96;    // splits per row a merge handles (context <= 96 blocks)
constexpr int kPhasesPerLayer = 9;
constexpr int kMaxCtaBlocks = 256;    // attention KV block ids a CTA keeps in shared memory
// phases of a layer (counter index 1 + 9 l + phase)
enum : int { kPhQKV = 0, kPhFinQ = 1, kPhAtt = 2, kPhO = 3, kPhFinO = 4, kPhGU = 6, kPhDown = 7, kPhFinD = 8 };
// Up to this many live rows the q/k/v and O projections are column-owned on warp-level MMAs
// (small_k), with their operand in fragment order.
constexpr int kSmallRows = 8;
constexpr int kSmallUnits = 2;  // 16-feature units a pass of small_k takes
constexpr int kSmallPhaseUnits = 2;   // QKV / O: units per participating CTA
constexpr int kCntStride = 16;        // phase counters 128 bytes apart (one L2 line each)
constexpr uint32_t kTmemCols = 512;
// Floats per head row of the attention states that a warp group joins in shared memory (128 dims,
// padded so that the eight heads' rows start in distinct banks).
constexpr int kAttORow = 132;
constexpr int kMinXBytes = kRingBytes - kMaxWSlots * kSlotBytes;
static_assert(2 * 4 * 8 * kAttORow * 4 <= kMinXBytes, "the joined attention states fit the X stages");
static_assert(8 * kSmallUnits * 16 * 8 * 4 <= kMinXBytes, "small_k's sums fit the X stages");
// Attention probabilities are taken against a running maximum that is re-based only when a
// score exceeds it by more than this (log2 units): P <= 2^8 in fp16, and most blocks skip the
// block maximum and the rescale of the output.
constexpr float kSoftmaxHeadroom = 8.f;

struct MegaParams {
    int layers, d, H, KVH, hd, F, V, Gq, nqkv;
    float eps, scale_log2;
    const uint8_t *w_qkv, *w_o, *w_gu, *w_down, *w_lm;  // blocked weights, layer strides below
    int64_t ls_qkv, ls_o, ls_gu, ls_down;
    const uint16_t *embed;                          // [V][d] bf16
    const uint16_t *attn_norm, *mlp_norm;           // [L][d]
    const uint16_t *final_norm;                     // [d]
    const float2 *rope;                             // [positions][hd/2] (cos, sin)
    uint8_t *kv;                                    // paged KV cache: block id b of layer l, kv head h
    int64_t kv_layer;                               // at kv + l * kv_layer + (b * KVH + h) * 64 KB
    StepPtrs c;
    int rows_cap, rows_cap16;
    int gp_qkv, gp_o;                               // CTAs taking part in the QKV / O projections
    float *x;                                       // [rows_cap][d] residual stream
    uint8_t *xg;                                    // pair-blocked [d/64][2 rows_cap16][64]
    uint8_t *att;                                   // pair-blocked [H*hd/64][2 rows_cap16][64]
    uint8_t *hm;                                    // pair-blocked [F/64][2 rows_cap16][64]
    float *ssqA, *ssqM;                             // [d/64][rows_cap] partial sums of x^2
    float *gpart;                                   // [segments][rows_cap][256] GEMM partial tiles
    uint16_t *qkv16;                                // [rows_cap][nqkv] fp16 q (scaled), k, v of the step
    float *part;                                    // [items][KVH][Gq][hd + 2] attention split partials
    int *att_cnt;                                   // [rows_cap][KVH] split arrival counters
    float *logits;                                  // [rows_cap][V] fp32, written if write_logits
    int write_logits;                               // teacher forcing: store the logits too
    unsigned long long *cnt;                        // phase arrival counters (monotonic), kCntStride apart
    unsigned long long *epoch;                      // launches completed since the reset
    uint64_t *stamps;                               // profiling builds: [cta][phase + 1][4] timestamps
    int n_stamp_ph;
    unsigned long long *ktime;                      // [2]: earliest CTA start, latest CTA end (ns)
};

// Profiling builds (-DSARA_STAMPS): per CTA and phase, when the compute warps arrived (0),
// when the phase's input dependency was observed (1), when the W producer finished issuing
// the phase's copies (2) and when the MMA issuer committed the phase's last MMA (3).
#ifdef SARA_STAMPS
#define MEGA_STAMP(ph, kind)                                                                              \
    do {                                                                                                  \
        if (p.stamps) p.stamps[((size_t)blockIdx.x * p.n_stamp_ph + (ph)) * 4 + (kind)] = globaltimer_ns(); \
    } while (0)
#else
#define MEGA_STAMP(ph, kind) \
    do {                     \
    } while (0)
#endif

// Attention unit: one split of one row for one kv head.  Split sp covers the `span` KV
// blocks from block sp * span on: positions [p0, p0 + n) of the row's ctx, in nb blocks.
struct AttUnit {
    int item, kvh, row, sp, ctx, p0, n, nb, nsplit, slot;
    int last;
};
constexpr int kMaxCtaUnits = 32;  // attention units a CTA keeps in shared memory

// A GEMM phase and this CTA's share of it (see SegWalk), fixed for a launch.
struct GemmPlan {
    const uint8_t *w, *x;  // blocked weights of layer 0, pair-blocked operand
    int64_t ls;            // bytes of a layer's weights
    int N, kch;            // output features, 64-column chunks of K
    int t, kc, units;      // first tile (16-feature unit) and chunk, units of this CTA
    int pass;              // column-owned: 16-feature units per pass; 0: split-K
};
constexpr int kPlanTiles = 32;  // contributor table entries per phase (wider phases compute them)

// W slots of a launch.  What the ring holds ahead is read while the step waits on a phase, so a fifth slot
// (5 MB over the CTAs) shortens the phases that stream weights; the activation stages give up its room,
// which costs more from 40 rows on, where a chunk takes 12 KB or more.  1.5B kernel, 4 -> 5 slots: one row
// of 100 positions 1.063 -> 1.043 ms, 16 rows 1.182 -> 1.148, 26 rows of 758 1.380 -> 1.352, 40 rows of
// 500 1.444 either way, 48 of 300 1.469 -> 1.474; the stages that need not be a power of two in
// number: 80 rows of 300 1.915 -> 1.885, 96 2.022 -> 1.977.
__host__ __device__ constexpr int ring_slots(int rows) { return rows <= 32 ? 5 : 4; }
// Bytes of an activation chunk (64 wide) in a stage: hi and lo parts of the rows' 8-row groups.
__host__ __device__ constexpr int x_chunk_bytes(int rows) { return rows <= 8 ? 2048 : (rows + 15) / 16 * 4096; }

struct MegaSmem {
    uint64_t wfull[kMaxWSlots], wempty[kMaxWSlots];
    uint64_t kvready[2][kMaxWSlots];  // attention: ring slot s holds warp group g's next KV tile
    uint64_t xfull[kMaxXStages], xempty[kMaxXStages];
    uint64_t acc_full[2], acc_empty[2];
    uint64_t drain;
    uint64_t units_ready;       // the attention unit table is filled (warp 0)
    unsigned long long target;  // counter value meaning "every CTA of this launch arrived"
    uint64_t wait_ns;           // bounded-wait limit of this launch
    float p_headroom;           // attention: log2 of how far P may exceed 1 before re-basing
    int stall_idx;              // test hook: the phase counter whose waits never complete (-1: none)
    uint32_t tmem_base;
    int abort;
    int rows, rows16, nws, nx, xgroup, xchunk, n_items, att_span;  // nws W slots; nx X stages of xgroup chunks
    GemmPlan plan[5];           // this CTA's share of each GEMM phase (the same for every layer)
    int2 tile_cta[3][kPlanTiles];  // first and last contributor of the tiles of q/k/v, O, down
    int small;                  // at most kSmallRows live rows
    float rstd[128];
    int rowpos[128];            // position of each live row
    // KV block ids: of this CTA's attention blocks (unit i's block j at ablk[aoff[i] + j]), and
    // of each row's current position (ablk_ok = 0: too many to hold, looked up in the table)
    AttUnit units[kMaxCtaUnits];
    AttUnit unit_tmp[kMegaThreads / 32][2];  // per warp: units beyond them, computed as they come
    int ablk[kMaxCtaBlocks];
    int aoff[kMaxCtaUnits];
    int rowblk[128];
    int ablk_ok;
    float red[2][4][8], red2[2][4][8];  // per warp group and warp: attention max / weighted sum of each head
    int kvrel[kMaxWSlots];                // warps that have read the slot's KV tile
    float mw[2][8][kMegaMaxSplits];      // per warp group: split weights of a merge
    float ml[2][8];
    int last_flag2[2];
};

// An MMA reads the operand rows of its M whether a chunk holds them or not (they feed accumulator rows that
// nobody reads): bytes past the last X stage's chunk, at most over the row counts.
__host__ __device__ constexpr int x_stage_chunks(int rows) { return rows <= 16 ? 4 : rows <= 32 ? 2 : 1; }
__host__ __device__ constexpr int x_stages(int rows) {
    const int n = (kRingBytes - ring_slots(rows) * kSlotBytes) / (x_chunk_bytes(rows) * x_stage_chunks(rows));
    return n < kMaxXStages ? n : kMaxXStages;
}
constexpr int x_overread() {
    int most = 0;
    for (int rows = 1; rows <= 128; ++rows) {
        const int operand = rows <= 32 ? 64 * 128 : rows <= 64 ? 128 * 128 : 2 * 128 * 128;
        const int end = ring_slots(rows) * kSlotBytes + (x_stages(rows) * x_stage_chunks(rows) - 1) * x_chunk_bytes(rows) + operand;
        most = end - kRingBytes > most ? end - kRingBytes : most;
    }
    return most;
}
static_assert(x_overread() <= (int)sizeof(MegaSmem), "the operands' don't-care rows stay inside the shared memory");
constexpr size_t kMegaSmemBytes = 1024 + (size_t)kRingBytes + sizeof(MegaSmem);
static_assert(kMegaSmemBytes <= 232448, "227 KB of shared memory per CTA");

// ------------------------------------------------------------------------------ layouts
// Pair-blocked activation (a GEMM operand held as bf16 hi + lo parts): per 64-wide k-chunk,
// 2 rows16 rows of 128 B (64 bf16, 128-byte swizzle) in 8-row groups that alternate between
// the hi parts of rows 8g..8g+7 and their lo parts.  Byte offset of the hi part of element
// (r, k); the lo part sits kLoOff bytes after it.  One MMA over the chunk's first 2 R16 rows
// multiplies hi and lo parts at once (rows16 <= 64); with a 2048-byte group stride the hi
// (lo) groups alone form a 128-row operand.
constexpr int kLoOff = 1024;
__host__ __device__ __forceinline__ uint32_t xblk_off(int r, int k, int rows16) {
    const int chunk = k >> 6, col = k & 63;
    return (uint32_t)(chunk * 2 * rows16 + 16 * (r >> 3) + (r & 7)) * 128 +
           ((((col >> 3) ^ (r & 7)) << 4) | ((col & 7) << 1));
}
// Fragment-order activation (the operand of small_k): per 32-wide k-block and 8-row tile, the hi
// then the lo part, each 32 lanes x 16 bytes: what lane 4 g + t of a warp needs of row g as
// m16n8k16 B fragments of the block's two k-steps, so a warp reads a (block, tile, part) with one
// coalesced 16-byte load per lane, straight into its registers.  Byte offset of the hi part of
// element (r, k); the lo part sits kFragLo after it.
constexpr int kFragLo = 512;
__host__ __device__ __forceinline__ uint32_t frag_off(int r, int k, int rows16) {
    return (uint32_t)((k >> 5) * (rows16 >> 3) + (r >> 3)) * 1024 + ((r & 7) * 4 + ((k & 7) >> 1)) * 16 +
           ((k >> 3) & 3) * 4 + (k & 1) * 2;
}
// Byte offsets of K(pp, d) and V(pp, d) inside one 128-position KV block.
__host__ __device__ __forceinline__ int kv_k_off(int pp, int d) {
    return (d >> 6) * 16384 + pp * 128 + (((((d & 63) >> 3) ^ (pp & 7)) << 4) | ((d & 7) << 1));
}
__host__ __device__ __forceinline__ int kv_v_off(int pp, int d) {
    const int c = pp & 63;
    return 32768 + (pp >> 6) * 16384 + d * 128 + ((((c >> 3) ^ (d & 7)) << 4) | ((c & 7) << 1));
}
// Order of a head's rows in the q/k/v weights: 16-row units of 8 dims of the first half and
// their rotation partners, the same dims of the second half.  Row of dim dd.
__host__ __device__ __forceinline__ int qkv_row(int dd, int half_hd) {
    const int i = dd < half_hd ? dd : dd - half_hd;
    return (i >> 3) * 16 + (i & 7) + (dd < half_hd ? 0 : 8);
}
// Byte offset of features col0.. (a multiple of 8) of k-chunk kc of a blocked weight matrix [N][K].
__device__ __forceinline__ int64_t wblk_off(int N, int col0, int kc) { return ((int64_t)kc * N + col0) * 128; }

// ------------------------------------------------------------------------------ waits
// The slow paths of the waits are functions of their own: inlined at every wait they made a third
// of the kernel's code, which does not fit the instruction cache as it is.
__device__ __noinline__ bool mwait_slow(uint32_t bar, uint32_t parity, int *err, volatile int *abort, uint64_t limit) {
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63u) == 0) {
            if (*abort) return false;
            if (globaltimer_ns() - t0 > limit) {
                report_error(err, ERR_WAIT_TIMEOUT);
                *abort = 1;
                return false;
            }
        }
    }
}
// Bounded mbarrier wait that also gives up (returning false) once the CTA is aborting.
__device__ __forceinline__ bool mwait(uint64_t *bar, uint32_t parity, int *err, volatile int *abort, uint64_t limit) {
    const uint32_t b = smem_u32(bar);
    if (mbar_try_wait(b, parity)) return true;
    return mwait_slow(b, parity, err, abort, limit);
}
// The same for a converged warp: one answer for all of its lanes.
__device__ __forceinline__ bool mwait_warp(uint64_t *bar, uint32_t parity, int *err, volatile int *abort, uint64_t limit) {
    const uint32_t b = smem_u32(bar);
    if (__all_sync(0xffffffffu, mbar_try_wait(b, parity))) return true;
    return __all_sync(0xffffffffu, mwait_slow(b, parity, err, abort, limit));
}

// Spin until a phase counter reaches `target` (acquire loads);
// bounded, gives up on abort or once another CTA reported a timeout.
__device__ __noinline__ bool spin_counter(const unsigned long long *cnt, unsigned long long target, int *err,
                                          volatile int *abort, uint64_t limit) {
    if (ld_acquire_u64(cnt) >= target) return true;
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t it = 1;; ++it) {
        __nanosleep(32);
        if (ld_acquire_u64(cnt) >= target) return true;
        if ((it & 15u) == 0) {
            if (*abort) return false;
            if (*(volatile int *)err & ERR_WAIT_TIMEOUT) {
                *abort = 1;
                return false;
            }
            if (globaltimer_ns() - t0 > limit) {
                report_error(err, ERR_WAIT_TIMEOUT);
                *abort = 1;
                return false;
            }
        }
    }
}
// The same for a converged warp: one lane polls.
__device__ __forceinline__ bool spin_counter_warp(const unsigned long long *cnt, unsigned long long target, int *err,
                                                  volatile int *abort, uint64_t limit) {
    bool r = false;
    if (elect_one()) r = spin_counter(cnt, target, err, abort, limit);
    return __any_sync(0xffffffffu, r);
}

// Counter value a wait on phase counter idx needs: every CTA of this launch arrived (the
// test hook makes one counter's target unreachable, so its waits run into the time limit).
__device__ __forceinline__ unsigned long long phase_target(const MegaParams &p, const MegaSmem &S, int idx) {
    return idx == S.stall_idx ? ~0ull : S.target;
}

// ------------------------------------------------------------------------------ phases
// GEMM phases: N output features, K inputs.  Two ways to split the work:
//   split-K: (256-feature tile, 64-column chunk) units in equal contiguous ranges over the CTAs;
//     each CTA stores its fp32 partial tiles and a finalisation phase sums them.
//   column-owned (gate / up; lm_head; q/k/v and O at few live rows): 16-feature units in equal contiguous
//     ranges, each with the whole K, so that the CTA's epilogue applies what follows (SwiGLU;
//     RoPE and the cache append; residual and norm input) itself and no partials and no
//     finalisation phase are needed.  More activation traffic (every CTA reads the whole
//     operand) and fewer weight rows per MMA, but one phase barrier and one L2 round trip less.
enum : int { kGQKV = 0, kGO = 1, kGDown = 2, kGGU = 3, kGLM = 4 };  // plan index
constexpr int kOwnCols = 16;  // features per unit of a column-owned phase
constexpr int kOwnUnits = kTileN / kOwnCols;  // units of a pass at most

// Geometry of a phase for CTA c of G: filled into plan[which] once per launch.
// (Unit counts stay below 2^31 / SMs for every supported shape: 32-bit products suffice.)
__device__ __noinline__ void make_plan(const MegaParams &p, GemmPlan &g, int which, int c, int G, bool small) {
    int K = p.d, Gp = G;
    g.x = p.xg;
    g.pass = 0;
    if (which == kGQKV) {
        g.w = p.w_qkv; g.ls = p.ls_qkv; g.N = p.nqkv; Gp = p.gp_qkv;
    } else if (which == kGO) {
        g.w = p.w_o; g.ls = p.ls_o; g.N = p.d; K = p.H * p.hd; g.x = p.att; Gp = p.gp_o;
    } else if (which == kGDown) {
        g.w = p.w_down; g.ls = p.ls_down; g.N = p.d; K = p.F; g.x = p.hm;
    } else if (which == kGGU) {
        g.w = p.w_gu; g.ls = p.ls_gu; g.N = 2 * p.F;
    } else {
        g.w = p.w_lm; g.ls = 0; g.N = p.V;
    }
    g.kch = K / 64;
    g.t = g.kc = g.units = 0;
    // at most one CTA per unit, so every participating CTA holds a
    // non-empty range and the CTAs between a tile's first and last owner all contributed
    const bool sm = small && (which == kGQKV || which == kGO);
    if (which == kGGU || which == kGLM || sm) {
        const int U = g.N / kOwnCols, most = sm ? kSmallUnits : kOwnUnits;
        Gp = min(G, U);
        if (sm) {  // equal shares: a pass of small_k costs about the same for one unit or two
            const int per = (U + Gp - 1) / Gp;
            Gp = (U + per - 1) / per;
        }
        if (c < Gp) {
            g.t = c * U / Gp;
            g.units = (c + 1) * U / Gp - g.t;
            if (which == kGLM && U >= kOwnUnits * 2 * Gp) {
                // a large vocabulary in whole passes: equal shares of 62.5 units read no faster
                // (1.5B, 151,936 tokens, 26 rows: 1.189 ms in tiles, 1.191 in shares)
                const int T = (U + kOwnUnits - 1) / kOwnUnits;
                g.t = c * T / Gp * kOwnUnits;
                g.units = min(U, (c + 1) * T / Gp * kOwnUnits) - g.t;
            }
            const int np = (g.units + most - 1) / most;  // equal passes
            g.pass = (g.units + np - 1) / np;
        }
    } else {
        const int U = (g.N + kTileN - 1) / kTileN * g.kch;
        Gp = min(Gp, U);
        if (c < Gp) {
            const int u0 = c * U / Gp;
            g.units = (c + 1) * U / Gp - u0;
            g.t = u0 / g.kch;
            g.kc = u0 - g.t * g.kch;
        }
    }
}

// A CTA's share of a phase walked as segments, each one accumulator: features [col0, col0 + n) x
// chunks [kc0, kc1), in weight ring slots of cps chunks each.
struct Seg {
    int t, col0, n, kc0, kc1, cps;
    __device__ __forceinline__ int entries() const { return (kc1 - kc0 + cps - 1) / cps; }
};
struct SegWalk {
    int t, kc, left;
    __device__ __forceinline__ SegWalk(const GemmPlan &g) : t(g.t), kc(g.kc), left(g.units) {}
    __device__ __forceinline__ bool next(const GemmPlan &g, Seg &s) {
        if (left <= 0) return false;
        s.t = t;
        if (g.pass > 0) {
            const int nu = min(g.pass, left);
            s.col0 = t * kOwnCols;
            s.n = nu * kOwnCols;
            s.kc0 = 0;
            s.kc1 = g.kch;
            t += nu;
            left -= nu;
        } else {
            const int m = min(left, g.kch - kc);
            s.col0 = t * kTileN;
            s.n = min(kTileN, g.N - s.col0);
            s.kc0 = kc;
            s.kc1 = kc + m;
            ++t;
            kc = 0;
            left -= m;
        }
        s.cps = 1 << (s.n > 128 ? 0 : s.n > 64 ? 1 : s.n > 32 ? 2 : s.n > 16 ? 3 : 4);
        return true;
    }
};
// CTA owning unit u when U units are cut into Gp equal contiguous ranges.
__device__ __forceinline__ int unit_owner(int u, int U, int Gp) {
    int c = u * Gp / U;
    while (c + 1 < Gp && (c + 1) * U / Gp <= u) ++c;
    while (c > 0 && c * U / Gp > u) --c;
    return c;
}
// First and last CTA holding a partial of tile t of a split-K phase.  CTA c's partial of tile t is
// segment c + t of the partial buffer (distinct for every (c, t) of a phase: ranges are ordered).
__device__ __noinline__ int2 tile_ctas(const MegaParams &p, const GemmPlan &g, int which, int t, int G) {
    const int U = (g.N + kTileN - 1) / kTileN * g.kch;
    const int Gp = min(which == kGQKV ? p.gp_qkv : which == kGO ? p.gp_o : G, U);
    return make_int2(unit_owner(t * g.kch, U, Gp), unit_owner((t + 1) * g.kch - 1, U, Gp));
}

// Unit a of the launch (written to shared memory: a struct returned by a function would go through
// local memory, whose lines the small L1 beside this kernel's shared memory does not keep).
__device__ __noinline__ void att_unit(const MegaParams &p, int a, int span, AttUnit *dst) {
    AttUnit u;
    u.item = a / p.KVH;
    u.kvh = a - u.item * p.KVH;
    const int2 it = __ldg(&p.c.att_items[u.item]);
    u.row = it.x;
    u.sp = it.y;
    u.ctx = __ldg(&p.c.row_pos[u.row]) + 1;
    u.p0 = u.sp * span * kKVPos;
    u.n = min(u.ctx - u.p0, span * kKVPos);
    u.nb = (u.n + kKVPos - 1) / kKVPos;
    u.nsplit = ((u.ctx + kKVPos - 1) / kKVPos + span - 1) / span;
    u.last = u.p0 + u.n == u.ctx;
    u.slot = __ldg(&p.c.row_slot[u.row]);
    *dst = u;
}
// Unit i of this CTA (the launch's unit a0 + i), for a converged warp; slot 0 / 1: which of the warp's
// own entries a unit beyond the table goes to.
__device__ __forceinline__ const AttUnit &cta_unit(const MegaParams &p, MegaSmem &S, int a0, int i, int slot) {
    if (S.ablk_ok) return S.units[i];
    AttUnit *t = &S.unit_tmp[threadIdx.x >> 5][slot];
    __syncwarp();
    if ((threadIdx.x & 31) == 0) att_unit(p, a0 + i, S.att_span, t);
    __syncwarp();
    return *t;
}

// Attention units in equal contiguous ranges, counted from the last CTA down: the QKV
// projection runs on the first CTAs, so a small unit count lands on CTAs that are free
// to prefetch during it.
__device__ __forceinline__ void att_range(const MegaParams &p, int n_items, int &a0, int &a1) {
    const int NU = n_items * p.KVH, G = (int)gridDim.x, v = G - 1 - (int)blockIdx.x;
    a0 = v * NU / G;
    a1 = (v + 1) * NU / G;
}
// Address of block id b, kv head h of layer l in the paged KV cache.
__device__ __forceinline__ uint8_t *kv_addr(const MegaParams &p, int l, int b, int h) {
    return p.kv + l * p.kv_layer + ((int64_t)b * p.KVH + h) * kKVBlockBytes;
}
// Block j of this CTA's attention unit ui (= a - a0) in layer l's KV cache.
__device__ __forceinline__ uint8_t *kv_block(const MegaParams &p, const MegaSmem &S, int l, const AttUnit &u, int ui,
                                             int j) {
    const int b = S.ablk_ok ? S.ablk[S.aoff[ui] + j]
                            : __ldg(&p.c.blk_tab[(int64_t)u.slot * p.c.nblk_max + u.p0 / kKVPos + j]);
    return kv_addr(p, l, b, u.kvh);
}

// The KV block ids of this CTA's attention units (one warp, lane i: unit a0 + i), read once
// per launch from the block table into shared memory for the W producer.
__device__ __forceinline__ void fill_att_blocks(const MegaParams &p, MegaSmem &S, int lane) {
    int a0, a1;
    att_range(p, S.n_items, a0, a1);
    const int nu = a1 - a0;
    bool ok = nu <= kMaxCtaUnits;
    int nb = 0, off = 0;
    if (ok) {
        if (lane < nu) {
            att_unit(p, a0 + lane, S.att_span, &S.units[lane]);
            nb = S.units[lane].nb;
        }
        int x = nb;  // inclusive warp scan of the block counts
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        off = x - nb;
        ok = __shfl_sync(0xffffffffu, x, 31) <= kMaxCtaBlocks;
    }
    if (ok && lane < nu) {
        S.aoff[lane] = off;
        const int32_t *src = p.c.blk_tab + (int64_t)S.units[lane].slot * p.c.nblk_max + S.units[lane].p0 / kKVPos;
        for (int j0 = 0; j0 < nb; j0 += 8) {  // eight loads in flight
            int v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = j0 + q < nb ? __ldg(src + j0 + q) : 0;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (j0 + q < nb) S.ablk[off + j0 + q] = v[q];
        }
    }
    if (lane == 0) S.ablk_ok = ok ? 1 : 0;
    __syncwarp();
}

// Slot of ring entry e: e mod nws (mul = 2^32 / nws rounded up: exact far beyond a launch's entries).
__device__ __forceinline__ uint32_t ring_slot(uint32_t e, uint32_t nws, uint32_t mul) { return e - __umulhi(e, mul) * nws; }

// Counter of a GEMM phase of layer l.
__device__ __forceinline__ int gemm_counter(int gk, int l) {
    return 1 + kPhasesPerLayer * l + (gk == kGQKV ? kPhQKV : gk == kGO ? kPhO : gk == kGGU ? kPhGU : kPhDown);
}

// ------------------------------------------------------------------------------ W producer
// GEMM phases in launch order: q/k/v, O, gate / up, down of every layer, then lm_head.
__device__ __forceinline__ int gemm_kind(int i) { return i == 0 ? kGQKV : i == 1 ? kGO : i == 2 ? kGGU : kGDown; }

__device__ __forceinline__ void mega_w_producer(const MegaParams &p, MegaSmem &S, uint8_t *sW) {
    volatile int *ab = &S.abort;
    const uint64_t lim = S.wait_ns;
    int *err = &p.c.v->err;
    const uint64_t pol = l2_policy_evict_first();
    const uint32_t nws = S.nws;
    uint32_t wi = 0, ws = 0, wpar = 0;  // ring entries so far, the next one's slot, parity of its round
    bool ok = true;
    auto acquire = [&]() -> bool { return wi < nws || mwait_warp(&S.wempty[ws], wpar ^ 1, err, ab, lim); };
    auto advance = [&]() {
        ++wi;
        if (++ws == nws) { ws = 0; wpar ^= 1; }
    };
    int a0, a1;
    att_range(p, S.n_items, a0, a1);
#pragma unroll 1
    for (int i = 0; i <= 4 * p.layers && ok; ++i) {
        const int l = i >> 2, gk = i == 4 * p.layers ? kGLM : gemm_kind(i & 3);
        const GemmPlan &g = S.plan[gk];
        const uint8_t *w = g.w + l * g.ls;
        const int64_t rowb = (int64_t)g.N * 128;  // bytes of a chunk
        SegWalk walk(g);
        Seg sg;
#pragma unroll 1
        while (ok && walk.next(g, sg)) {
            const uint32_t cb = (uint32_t)sg.n * 128;  // a chunk's bytes
            const uint8_t *src = w + sg.kc0 * rowb + (int64_t)sg.col0 * 128;
#pragma unroll 1
            for (int kc = sg.kc0; kc < sg.kc1; kc += sg.cps) {
                if (!acquire()) { ok = false; break; }
                const int s = (int)ws, m = min(sg.cps, sg.kc1 - kc);
                if (elect_one()) {
                    mbar_arrive_expect_tx(&S.wfull[s], (uint32_t)m * cb);
#pragma unroll 1
                    for (int j = 0; j < m; ++j, src += rowb)
                        bulk_load(sW + (size_t)s * kSlotBytes + (size_t)j * cb, src, cb, &S.wfull[s], pol);
                }
                src = w + (kc + m) * rowb + (int64_t)sg.col0 * 128;
                advance();
            }
        }
        MEGA_STAMP(gk == kGLM ? 1 + kPhasesPerLayer * l : gemm_counter(gk, l), 2);
        if (gk == kGQKV && ok) {
            // the attention phase's KV blocks follow the QKV weights in ring order: unit
            // pairs (one unit per compute warp group), block by block, the K of the pair's
            // units, then their V^T; each one ring entry (K: d < 64 | d >= 64 halves, V^T:
            // positions < 64 | >= 64).  None depends on this step: the new position's k and v are
            // put into the tiles, and into the cache, by the warp that reads them.
#pragma unroll 1
            for (int a = a0; a < a1 && ok; a += 2) {
                const bool two = a + 1 < a1;
                const AttUnit &ua = cta_unit(p, S, a0, a - a0, 0);
                const AttUnit &ub = two ? cta_unit(p, S, a0, a - a0 + 1, 1) : ua;
                const int nbb = two ? ub.nb : 0, nbm = max(ua.nb, nbb);
#pragma unroll 1
                for (int q = 0; q < 4 * nbm && ok; ++q) {  // block q / 4, K or V^T, unit a or a + 1
                    const int j = q >> 2, kv = (q >> 1) & 1, x = q & 1;
                    if (j >= (x ? nbb : ua.nb)) continue;
                    const int n = x ? ub.n : ua.n;
                    const uint8_t *blk = kv_block(p, S, l, x ? ub : ua, a - a0 + x, j) + kv * 32768;
                    const int nj = min(kKVPos, n - j * kKVPos);
                    if (!acquire()) { ok = false; break; }
                    const int s = (int)ws;
                    // K: rows = positions, halves of the dims; V^T: rows = dims, halves of the positions
                    const uint32_t hb = kv == 0 ? (uint32_t)(((nj + 7) & ~7) * 128) : (uint32_t)(p.hd * 128);
                    const bool both = kv == 0 ? p.hd > 64 : nj > 64;
                    if (elect_one()) {
                        mbar_arrive_expect_tx(&S.wfull[s], both ? 2 * hb : hb);
                        bulk_load(sW + (size_t)s * kSlotBytes, blk, hb, &S.wfull[s], pol);
                        if (both) bulk_load(sW + (size_t)s * kSlotBytes + 16384, blk + 16384, hb, &S.wfull[s], pol);
                    }
                    advance();
                }
            }
            MEGA_STAMP(1 + kPhasesPerLayer * l + kPhAtt, 2);
        }
    }
    if (!ok) {  // every copy already issued lands before the CTA exits
        for (uint32_t s = 0; s < nws && s < wi; ++s) {
            const uint32_t last = (wi - 1 - s) / nws;  // round of its last use
            mbar_wait(&S.wfull[s], last & 1, err);
        }
    }
}

// ------------------------------------------------------------------------------ X producer
__device__ __forceinline__ void mega_x_producer(const MegaParams &p, MegaSmem &S, uint8_t *sX) {
    volatile int *ab = &S.abort;
    const uint64_t lim = S.wait_ns;
    int *err = &p.c.v->err;
    const uint64_t pol = l2_policy_evict_last();
    const int NX = S.nx, gx = S.xgroup;
    const uint32_t chunk = (uint32_t)S.xchunk;  // hi + lo parts of the live rows' groups
    const uint32_t stage = (uint32_t)gx * chunk;
    const int64_t chunk_stride = (int64_t)p.rows_cap16 * 256;
    uint32_t xi = 0;
    int xs = 0;          // the next stage
    uint32_t xpar = 0;   // parity of its round
    bool ok = true;
#pragma unroll 1
    for (int i = 0; i <= 4 * p.layers && ok; ++i) {
        const int l = i >> 2, gk = i == 4 * p.layers ? kGLM : gemm_kind(i & 3);
        const GemmPlan &g = S.plan[gk];
        SegWalk walk(g);
        if (walk.left <= 0 || (S.small && (gk == kGQKV || gk == kGO))) continue;  // (small_k loads its own)
        // the phase this operand comes from: FIN_D of l-1 / embedding, ATT, FIN_O, GU
        const int dep = kPhasesPerLayer * l + (gk == kGO ? 1 + kPhAtt : gk == kGGU ? 1 + kPhFinO : gk == kGDown ? 1 + kPhGU : 0);
        if (!spin_counter_warp(&p.cnt[dep * kCntStride], phase_target(p, S, dep), err, ab, lim)) { ok = false; break; }
        MEGA_STAMP(gk == kGLM ? 1 + kPhasesPerLayer * l : gemm_counter(gk, l), 1);
        fence_proxy_async_global();
        Seg sg;
#pragma unroll 1
        while (ok && walk.next(g, sg)) {
            const uint8_t *src = g.x + sg.kc0 * chunk_stride;
#pragma unroll 1
            for (int kc = sg.kc0; kc < sg.kc1; kc += gx, ++xi) {
                const int s = xs, m = min(gx, sg.kc1 - kc);
                if (xi >= (uint32_t)NX && !mwait_warp(&S.xempty[s], xpar ^ 1, err, ab, lim)) { ok = false; break; }
                if (elect_one()) {
                    mbar_arrive_expect_tx(&S.xfull[s], (uint32_t)m * chunk);
#pragma unroll 1
                    for (int j = 0; j < m; ++j)
                        bulk_load(sX + (size_t)s * stage + (size_t)j * chunk, src + j * chunk_stride, chunk, &S.xfull[s], pol);
                }
                src += gx * chunk_stride;
                if (++xs == NX) { xs = 0; xpar ^= 1; }
            }
        }
    }
    if (!ok) {
        for (uint32_t s = 0; s < (uint32_t)NX && s < xi; ++s) {
            const uint32_t last = (xi - 1 - s) / (uint32_t)NX;  // round of its last use
            mbar_wait(&S.xfull[s], last & 1, err);
        }
    }
}

// ------------------------------------------------------------------------------ MMA issuer
__device__ __forceinline__ void mega_mma(const MegaParams &p, MegaSmem &S, uint8_t *sW, uint8_t *sX, uint32_t tmem) {
    volatile int *ab = &S.abort;
    const uint64_t lim = S.wait_ns;
    int *err = &p.c.v->err;
    const int NX = S.nx, R16 = S.rows16, gx = S.xgroup;
    const uint32_t chunk = (uint32_t)S.xchunk, stage = (uint32_t)gx * chunk;
    // at most 64 live rows: one MMA per k-step over the stacked hi / lo groups (M = 2 R16
    // rounded up to 64 or 128: the rows past the stage only feed accumulator rows nobody
    // reads); more: the hi and the lo groups as two 128-row operands into one accumulator
    const bool stacked = R16 <= 64;
    const uint32_t sbo = stacked ? 1024u : 2048u;
    uint32_t ws = 0, wpar = 0, xs = 0, xpar = 0;  // the next W slot / X stage and the parity of its round
    uint32_t use[2] = {0, 0};  // accumulator buffer uses
    uint32_t tseg = 0;         // segments so far
    bool ok = true;
    const uint32_t nws = S.nws;
    auto w_advance = [&]() {
        if (++ws == nws) { ws = 0; wpar ^= 1; }
    };
    int a0, a1;
    att_range(p, S.n_items, a0, a1);
    int gi = 0;  // attention units so far (unit i of a phase runs on group (gi + i) & 1)
#pragma unroll 1
    for (int i = 0; i <= 4 * p.layers && ok; ++i) {
        const int gk = i == 4 * p.layers ? kGLM : gemm_kind(i & 3);
        const GemmPlan &g = S.plan[gk];
        SegWalk walk(g);
        Seg sg;
        const bool fwd = S.small && (gk == kGQKV || gk == kGO);
#pragma unroll 1
        while (ok && walk.next(g, sg)) {
            if (fwd) {  // small_k's weights: handed over to both compute groups as they land (see below)
#pragma unroll 1
                for (int e = sg.entries(); e > 0; --e) {
                    if (!mwait_warp(&S.wfull[ws], wpar, err, ab, lim)) { ok = false; break; }
                    if (elect_one()) {
                        mbar_arrive(&S.kvready[0][ws]);
                        mbar_arrive(&S.kvready[1][ws]);
                    }
                    w_advance();
                }
                continue;
            }
            const uint32_t a = tseg & 1;  // segments alternate between two accumulators (epilogue overlaps)
            const uint32_t use_a = a ? use[1] : use[0];
            if (use_a >= 1 && !mwait_warp(&S.acc_empty[a], (use_a - 1) & 1, err, ab, lim)) { ok = false; break; }
            tc_fence_after();
            const uint32_t d = tmem + a * kTileN;
            const uint32_t idg = idesc_bf16_f32(R16 <= 32 ? 64u : 128u, (uint32_t)sg.n);
            const uint32_t cb = (uint32_t)sg.n * 128;
            // chunks go in groups that stay within one weight slot and one activation stage, so a
            // group's MMAs issue back to back: one pair of waits and commits per group
            const int grp = min(sg.cps, gx);
            int wj = 0, xj = 0;  // chunk within the weight slot / the activation stage
#pragma unroll 1
            for (int kc = sg.kc0; kc < sg.kc1; kc += grp) {
                if (wj == 0 && !mwait_warp(&S.wfull[ws], wpar, err, ab, lim)) { ok = false; break; }
                if (xj == 0 && !mwait_warp(&S.xfull[xs], xpar, err, ab, lim)) { ok = false; break; }
                tc_fence_after();
                const int m = min(grp, sg.kc1 - kc);
                const bool end = kc + m == sg.kc1;
                const bool wlast = end || wj + grp == sg.cps, xlast = end || xj + grp == gx;
                if (elect_one()) {
                    uint32_t aw = smem_u32(sW) + ws * kSlotBytes + (uint32_t)wj * cb;
                    uint32_t ax = smem_u32(sX) + xs * stage + (uint32_t)xj * chunk;
                    uint32_t acc = kc == sg.kc0 ? 0u : 1u;
#pragma unroll 1
                    for (int j = 0; j < m; ++j, aw += cb, ax += chunk) {
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            const uint64_t bd = sdesc_kmajor_sw128(aw + kk * 32);
                            tc_mma_bf16(d, sdesc_kmajor_sw128(ax + kk * 32, sbo), bd, idg, acc);
                            acc = 1u;
                            if (!stacked) tc_mma_bf16(d, sdesc_kmajor_sw128(ax + kLoOff + kk * 32, sbo), bd, idg, 1u);
                        }
                    }
                    if (xlast) tc_commit(&S.xempty[xs]);
                    if (wlast) tc_commit(&S.wempty[ws]);
                    if (end) tc_commit(&S.acc_full[a]);
                }
                __syncwarp();
                wj = wlast ? 0 : wj + grp;
                xj = xlast ? 0 : xj + grp;
                if (wlast) w_advance();
                if (xlast && ++xs == (uint32_t)NX) { xs = 0; xpar ^= 1; }
            }
            if (a) ++use[1]; else ++use[0];
            ++tseg;
        }
        MEGA_STAMP(gk == kGLM ? 1 + kPhasesPerLayer * (i >> 2) : gemm_counter(gk, i >> 2), 3);
        if (gk == kGQKV && ok) {
            // The attention phase's ring entries (its KV tiles) are read and released by the compute
            // warp groups.  The issuer is the ring's one in-order observer: it waits for each entry to
            // land and hands it to the group that runs its unit (an arrival on kvready[group][slot]).
            // A group's consecutive uses of a slot are then at most one barrier phase apart (the slot
            // is refilled only after the group released its previous tile there), which a group
            // waiting on the shared wfull barriers directly could not rely on.
            const int n = a1 - a0;
            if (i == 0 && !mwait_warp(&S.units_ready, 0, err, ab, lim)) ok = false;
#pragma unroll 1
            for (int u = 0; u < n && ok; u += 2) {
                const bool two = u + 1 < n;
                const int nba = cta_unit(p, S, a0, u, 0).nb, nbb = two ? cta_unit(p, S, a0, u + 1, 1).nb : 0;
                const int nbm = max(nba, nbb);
#pragma unroll 1
                for (int q = 0; q < 4 * nbm; ++q) {  // the W producer's order
                    const int j = q >> 2, x = q & 1;
                    if (j >= (x ? nbb : nba)) continue;
                    if (!mwait_warp(&S.wfull[ws], wpar, err, ab, lim)) { ok = false; break; }
                    if (elect_one()) mbar_arrive(&S.kvready[(gi + u + x) & 1][ws]);
                    w_advance();
                }
            }
            gi += n;
            MEGA_STAMP(1 + kPhasesPerLayer * (i >> 2) + kPhAtt, 3);
        }
    }
    // every MMA issued has retired before tensor memory is released
    if (elect_one()) tc_commit(&S.drain);
    mbar_wait(&S.drain, 0, err);
}

// ------------------------------------------------------------------------------ compute
// Column-owned projection of up to 8 rows on warp-level MMAs: sum_k W[c][k] X[r][k] for the
// segment's one or two 16-feature units, the whole K split over the eight compute warps by
// 32-wide k-blocks (block kb on warp kb % 8).  X comes straight from global memory in fragment
// order (three blocks' loads in flight at once), W from the ring's slots, which the issuer hands
// over; the per-warp sums go to red[warp][unit][feature][row rotated by feature].
// Against the split-K tcgen05 phase plus its finalisation phase this is one phase barrier and
// two L2 round trips less (q/k/v at one row: 7.3 -> 5.0 us per layer, O: 6.8 -> 4.5); every CTA
// reads the whole operand, so above 8 rows the gain is gone (26 rows: 16.5 -> 14.2 us for both,
// but as much lost to the larger code of the other phases).
template <typename KvWait>
__device__ __forceinline__ void small_k(MegaSmem &S, const uint8_t *sW, float *red, const uint8_t *X, int rows16, int kch,
                                        const Seg &sg, uint32_t wring, int cw, int lane, KvWait &&kv_wait, uint32_t nws_mul) {
    constexpr int B = 3;  // k-blocks per batch (more would spill registers, in every phase of the kernel)
    const int mt = sg.n / kOwnCols, E = sg.entries(), lgc = __ffs(sg.cps) - 1;
    const uint32_t kbs = (uint32_t)(rows16 >> 3) * 1024;  // bytes of a k-block
    float acc[kSmallUnits][4];
#pragma unroll
    for (int m = 0; m < kSmallUnits; ++m)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[m][q] = 0.f;
    const int arow = lane & 15;  // ldmatrix row of this lane
#pragma unroll 1
    for (int e0 = 0; e0 < E; e0 += S.nws) {  // as many slots as the ring holds
        const int e1 = min(E, e0 + S.nws);
        const int kb1 = min(2 * kch, 2 * sg.cps * e1);
        int seen = e0;  // slots handed over so far
#pragma unroll 1
        for (int kb0 = 2 * sg.cps * e0 + cw; kb0 < kb1; kb0 += 8 * B) {
            uint4 xh[B], xl[B];
            const uint8_t *src = X + kb0 * kbs + lane * 16;
#pragma unroll
            for (int b = 0; b < B; ++b, src += 8 * kbs) {
                xh[b] = xl[b] = make_uint4(0, 0, 0, 0);
                if (kb0 + 8 * b < kb1) {
                    xh[b] = __ldcg(reinterpret_cast<const uint4 *>(src));
                    xl[b] = __ldcg(reinterpret_cast<const uint4 *>(src + kFragLo));
                }
            }
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int kb = kb0 + 8 * b;
                if (kb < kb1) {
                    const int e = (kb >> 1) >> lgc;
#pragma unroll 1
                    for (; seen <= e; ++seen) kv_wait(wring + seen);
                    const uint32_t wb = smem_u32(sW) + ring_slot(wring + e, S.nws, nws_mul) * kSlotBytes +
                                        (uint32_t)(((kb >> 1) - (e << lgc)) * sg.n * 128 + arow * 128);
#pragma unroll
                    for (int ks = 0; ks < 2; ++ks) {
                        const int gran = ((kb & 1) * 2 + ks) * 2 + (lane >> 4);
#pragma unroll
                        for (int m = 0; m < kSmallUnits; ++m) {
                            if (m < mt) {
                                uint32_t a[4];
                                ldsm_x4(wb + m * kOwnCols * 128 + ((gran ^ (arow & 7)) << 4), a);
                                mma_bf16_16816(acc[m], a, ks ? xh[b].z : xh[b].x, ks ? xh[b].w : xh[b].y);
                                mma_bf16_16816(acc[m], a, ks ? xl[b].z : xl[b].x, ks ? xl[b].w : xl[b].y);
                            }
                        }
                    }
                }
            }
        }
#pragma unroll 1
        for (; seen < e1; ++seen) kv_wait(wring + seen);  // (every thread follows every hand-over)
        if (e1 < E) {
            named_bar_sync(1, kMegaCThreads);
            if (cw == 0 && lane == 0)
                for (int e = e0; e < e1; ++e) mbar_arrive(&S.wempty[ring_slot(wring + e, S.nws, nws_mul)]);
        }
    }
#pragma unroll
    for (int m = 0; m < kSmallUnits; ++m)
        if (m < mt) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int c = (lane >> 2) + 8 * (q >> 1), r = 2 * (lane & 3) + (q & 1);
                red[((cw * kSmallUnits + m) * kOwnCols + c) * 8 + ((r + c) & 7)] = acc[m][q];
            }
        }
}

// The compute warps' code runs once per layer and is far larger than the instruction caches'
// first levels, so its size is time: each step exists once (the layer loop is unrolled over
// nothing, the three residual finalisations and the three split-K epilogues share their code),
// divisions by launch constants are done once (GemmPlan, tile_cta), and batches of loads are
// spread over the lanes instead of being unrolled further.
__device__ __forceinline__ void mega_compute(const MegaParams &p, MegaSmem &S, uint8_t *sW, uint8_t *sX, uint32_t tmem) {
    volatile int *ab = &S.abort;
    const uint64_t lim = S.wait_ns;
    int *err = &p.c.v->err;
    const int ctid = threadIdx.x - 96;  // 0..255
    const int cw = ctid >> 5, lane = threadIdx.x & 31;
    const int quarter = (threadIdx.x >> 5) & 3;  // tensor-memory lanes 32*quarter ..
    const int half = cw >> 2;                    // warps 3..6 -> 0, 7..10 -> 1
    const int G = gridDim.x, cta = blockIdx.x;
    const int R = S.rows, R16c = p.rows_cap16;
    const bool small = S.small != 0;
    const int d = p.d, hd = p.hd, Gq = p.Gq;
    const int gw = cta * 8 + cw, nw = G * 8;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    // GEMM accumulator lane -> activation row.  Stacked operand (at most 64 live rows): operand
    // row m holds the hi (lo) part of row 8 (m / 16) + m % 8 for m % 16 < 8 (>= 8); M = 128
    // puts operand row m in lane m, M = 64 (at most 32 rows) in lane 32 (m / 16) + m % 16.
    // The hi and lo accumulators of a row are lanes i and i ^ 8 of one warp: after adding them
    // with a shuffle each lane of the pair finishes half of the columns.  Otherwise (M = 128,
    // hi and lo accumulated together) row i is lane i.  Lanes of no row: past the batch.
    const int R16 = S.rows16;
    const bool pair = R16 <= 64, second = pair && (lane & 8) != 0;
    const int my_row = R16 <= 32 ? ((lane & 16) == 0 ? quarter * 8 + (lane & 7) : 1 << 20)
                       : pair    ? quarter * 16 + 8 * (lane >> 4) + (lane & 7)
                                 : quarter * 32 + lane;
    const bool act = my_row < R;
    const bool quarter_live = (R16 <= 32 ? quarter * 8 : pair ? quarter * 16 : quarter * 32) < R;
    uint32_t wring = 0;  // W ring entries of the phases before the current one (the producer's count)
    uint32_t kvpar = 0;  // per ring slot (bit s): parity of this warp group's next kvready wait
    const uint32_t nws = S.nws, nws_mul = 0xffffffffu / nws + 1;
    auto wslot = [&](uint32_t e) { return ring_slot(e, nws, nws_mul); };
    auto kv_wait = [&](uint32_t e) {
        const uint32_t sl = wslot(e);
        mwait(&S.kvready[half][sl], (kvpar >> sl) & 1u, err, ab, lim);
        kvpar ^= 1u << sl;
    };
    int gi = 0;             // attention units so far
    uint32_t cuse = 0;      // bit a: parity of accumulator a's next use
    uint32_t tseg = 0;      // GEMM segments so far
    auto acc_wait = [&]() -> uint32_t {  // the next segment's accumulator, its MMAs done
        const uint32_t a = tseg & 1;
        mwait(&S.acc_full[a], (cuse >> a) & 1u, err, ab, lim);
        tc_fence_after();
        return a;
    };
    auto acc_release = [&](uint32_t a) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.acc_empty[a]);
        cuse ^= 1u << a;
        ++tseg;
    };
    // What the other lane of a pair holds of this lane's 16 of 32 columns (not a pair: nothing).
    auto pair_part = [&](const float (&v)[32], float (&w)[16]) {
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const float t = __shfl_xor_sync(0xffffffffu, second ? v[e] : v[16 + e], 8);
            w[e] = pair ? t : 0.f;
        }
    };
    // phase arrival: the CTA's writes of this phase (made visible to thread 0 by the barrier)
    // are released to the other CTAs with the counter increment
    // (x_operand: this phase wrote a GEMM operand that bulk copies of other CTAs will read)
    auto arrive = [&](int idx, bool x_operand) {
        if (x_operand) fence_proxy_async_global();
        named_bar_sync(1, kMegaCThreads);
        if (ctid == 0) {
            MEGA_STAMP(idx, 0);
            red_add_release_gpu(&p.cnt[idx * kCntStride], 1ull);
        }
    };
    auto wait_phase = [&](int idx) {
        if (ctid == 0) {
            spin_counter(&p.cnt[idx * kCntStride], phase_target(p, S, idx), err, ab, lim);
            MEGA_STAMP(idx + 1, 1);
        }
        named_bar_sync(1, kMegaCThreads);
    };
    // 1/rms of every row from its np (at most 128) partial sums of squares: a warp per row, a
    // lane per partial
    auto load_rstd = [&](const float *ssq, int np) {
#pragma unroll 1
        for (int r = cw; r < R; r += 8) {
            float s = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (lane + 32 * q < np) s += __ldcg(&ssq[(lane + 32 * q) * p.rows_cap + r]);
            s = warp_sum(s);
            if (lane == 0) S.rstd[r] = rsqrtf(s / (float)d + p.eps);
        }
    };
    // contributors of tile t of split-K phase `which`
    auto contributors = [&](int which, int t) -> int2 {
        return t < kPlanTiles ? S.tile_cta[which][t] : tile_ctas(p, S.plan[which], which, t, G);
    };
    // Four columns' sum of a tile's partials for one row.  split: lanes 0-15 and 16-31 of a warp have
    // the same columns, take alternate contributors (up to 16 loads in flight each), then add up.
    // `off`: row and column inside a segment, in floats.
    auto part_sum = [&](int2 ct, int t, int off, bool split) -> float4 {
        const int64_t seg = (int64_t)p.rows_cap * kTileN;
        const int c0 = split ? lane >> 4 : 0;
        const int64_t step = split ? 2 * seg : seg;
        const float *src = p.gpart + (int64_t)(ct.x + c0 + t) * seg + off;
        int n = split ? (ct.y - ct.x - c0 + 2) >> 1 : ct.y - ct.x + 1;  // contributors of this lane
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
        while (__any_sync(0xffffffffu, n > 0)) {
            float4 v[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (k < n) v[k] = __ldcg(reinterpret_cast<const float4 *>(src));
                src += step;
            }
#pragma unroll
            for (int k = 0; k < 16; ++k) { s.x += v[k].x; s.y += v[k].y; s.z += v[k].z; s.w += v[k].w; }
            n -= 16;
        }
        if (!split) return s;
        s.x += __shfl_xor_sync(0xffffffffu, s.x, 16);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, 16);
        s.z += __shfl_xor_sync(0xffffffffu, s.z, 16);
        s.w += __shfl_xor_sync(0xffffffffu, s.w, 16);
        return s;
    };

    // the attention output's layout: the O projection's operand
    auto att_off = [&](int r, int kk) -> uint32_t { return small ? frag_off(r, kk, R16c) : xblk_off(r, kk, R16c); };
    const int lo_off = small ? kFragLo : kLoOff;

    // the KV block of each row's current position (its k, v are appended there every layer)
    if (ctid < R) {
        const int pos = __ldg(&p.c.row_pos[ctid]);
        S.rowpos[ctid] = pos;
        S.rowblk[ctid] = __ldg(&p.c.blk_tab[(int64_t)__ldg(&p.c.row_slot[ctid]) * p.c.nblk_max + pos / kKVPos]);
    }

    // Steps 3 l + k of layer l: k = 0: residual and attention norm input (embedding, or the
    // previous layer's down projection), then the q/k/v GEMM; 1: q, k, v and attention, then the
    // O GEMM; 2: residual and MLP norm input, gate / up, then the down GEMM.  Step 3 L ends with
    // the final norm input.
#pragma unroll 1
    for (int step = 0, l = 0, k = 0;; ++step) {
        const int base = 1 + kPhasesPerLayer * l;
        const bool fin = k == 0 || (k == 2 && !small);
        if (fin) {
            // ---------------------------------------------------- residual, next norm input
            // x += sum of the GEMM's partials (x = E[tok] at the start); x_g = x * gn as a blocked
            // hi/lo pair; per (row, 64 features) sum of squares.  Unit = (row, 64 features): lane
            // % 16 = 4 features.  While no warp has more than one unit its two halves split the
            // contributors, then the first stores x and the hi parts, the second the lo parts; above,
            // a half warp takes a unit, so that fewer of them follow one another in a warp.  Kernel,
            // ms with split units -> with half warps: 1.5B 48 rows of 60 positions (one unit) 1.317 ->
            // 1.332, 64 rows (two) 1.439 -> 1.395, 100 rows 1.806 -> 1.761; 3B 48 rows 2.212 -> 2.147.
            const int which = k == 0 ? kGDown : kGO;
            const uint16_t *gn = k == 2 ? p.mlp_norm + l * d : l < p.layers ? p.attn_norm + l * d : p.final_norm;
            float *ssq = k == 2 ? p.ssqM : p.ssqA;
            if (step > 0) wait_phase(k == 2 ? base + kPhO : base - kPhasesPerLayer + kPhDown);
            const int d64 = d / 64, nu = R * d64;
            const bool split = small || nu <= nw;
            const int per = split ? 1 : 2, add = split ? 0 : lane >> 4;  // units of a warp, of which this lane's
#pragma unroll 1
            for (int u0 = per * gw; u0 < nu; u0 += per * nw) {
                const bool own = u0 + add < nu;
                const int u = own ? u0 + add : u0;
                const int r = u / d64, h64 = u - r * d64;
                const int f = h64 * 64 + (lane & 15) * 4;
                // the norm weights load with the residual and the partials
                const uint2 gb = __ldg(reinterpret_cast<const uint2 *>(gn + f));
                float4 x;
                float *xp = p.x + r * d + f;
                if (step == 0) {
                    int tok = p.c.row_tok[r];
                    if (tok < 0 || tok >= p.V) {
                        if ((lane & 15) == 0) report_error(err, ERR_BOUNDS);
                        tok = 0;
                    }
                    const uint2 e = __ldg(reinterpret_cast<const uint2 *>(p.embed + (int64_t)tok * d + f));
                    x = make_float4(bf16_to_f32(e.x & 0xffff), bf16_to_f32(e.x >> 16), bf16_to_f32(e.y & 0xffff),
                                    bf16_to_f32(e.y >> 16));
                } else {
                    x = __ldcg(reinterpret_cast<const float4 *>(xp));
                    const int t = f / kTileN;
                    const float4 s = part_sum(contributors(which, t), t, r * kTileN + f - t * kTileN, split);
                    x.x += s.x; x.y += s.y; x.z += s.z; x.w += s.w;
                }
                uint16_t h[4], lo[4];
                split_bf16(x.x * bf16_to_f32(gb.x & 0xffff), h[0], lo[0]);
                split_bf16(x.y * bf16_to_f32(gb.x >> 16), h[1], lo[1]);
                split_bf16(x.z * bf16_to_f32(gb.y & 0xffff), h[2], lo[2]);
                split_bf16(x.w * bf16_to_f32(gb.y >> 16), h[3], lo[3]);
                const bool first = lane < 16 || !split;  // stores x (and the hi parts)
                float sq = first ? (x.x * x.x + x.y * x.y) + (x.z * x.z + x.w * x.w) : 0.f;
                if (first && own) *reinterpret_cast<float4 *>(xp) = x;
                const uint2 w = first ? pack4(h) : pack4(lo);
                if (small && l < p.layers) {  // small_k's operand
                    uint8_t *dst = p.xg + frag_off(r, f, R16c) + (first ? 0 : kFragLo);
                    *reinterpret_cast<uint32_t *>(dst) = w.x;
                    *reinterpret_cast<uint32_t *>(dst + 16) = w.y;
                } else if (own) {
                    uint8_t *dst = p.xg + xblk_off(r, f, R16c);
                    *reinterpret_cast<uint2 *>(dst + (first ? 0 : kLoOff)) = w;
                    if (!split) *reinterpret_cast<uint2 *>(dst + kLoOff) = pack4(lo);
                }
#pragma unroll
                for (int o2 = 8; o2 > 0; o2 >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o2);
                if ((lane & 15) == 0 && first && own) ssq[h64 * p.rows_cap + r] = sq;
            }
            arrive(k == 2 ? base + kPhFinO : base - 1, true);
            if (l == p.layers) break;
        }
        if (k == 2) {
            {
                // ------------------------------------------------ gate / up with SwiGLU
                // h = silu(r g) * (r u) straight from the accumulator: this CTA's features hold the
                // whole K, in 16-feature units of 8 gate then 8 up features.  The two warp halves
                // take alternate pairs of units; each lane of a pair finishes one unit of its row.
                // The row's 1/rms is read while the MMAs run.
                wait_phase(base + kPhFinO);
                load_rstd(p.ssqM, small ? d / kOwnCols : d / 64);
                named_bar_sync(1, kMegaCThreads);
                const float rs = act ? S.rstd[my_row] : 0.f;
                const GemmPlan &g = S.plan[kGGU];
                SegWalk walk(g);
                Seg sg;
#pragma unroll 1
                while (walk.next(g, sg)) {
                    wring += (uint32_t)sg.entries();
                    const uint32_t a = acc_wait();
                    const int nu = sg.n / kOwnCols;
                    if (quarter_live) {
#pragma unroll 1
                        for (int un = 2 * half; un < nu; un += 4) {
                            float v[32];
                            tmem_ld_32x32b_x32(tmem + lane_base + a * kTileN + un * kOwnCols, v);
                            float w[16];
                            pair_part(v, w);
#pragma unroll 1
                            for (int q = second ? 1 : 0; q < (pair && !second ? 1 : 2); ++q) {
                                if (!act || un + q >= nu) continue;
                                uint16_t hh[8], hl[8];
#pragma unroll
                                for (int e = 0; e < 8; ++e) {
                                    const float gv = ((q ? v[16 + e] : v[e]) + w[e]) * rs;
                                    const float uv = ((q ? v[24 + e] : v[8 + e]) + w[8 + e]) * rs;
                                    split_bf16(gv / (1.0f + expf(-gv)) * uv, hh[e], hl[e]);
                                }
                                uint8_t *dst = p.hm + xblk_off(my_row, sg.col0 / 2 + (un + q) * 8, R16c);
                                *reinterpret_cast<uint4 *>(dst) = pack8(hh);
                                *reinterpret_cast<uint4 *>(dst + kLoOff) = pack8(hl);
                            }
                        }
                    }
                    acc_release(a);
                }
                arrive(base + kPhGU, true);
            }
        } else if (k == 1) {
            int a0, a1;
            att_range(p, S.n_items, a0, a1);
            const int n = a1 - a0;
            if (l == 0) mwait(&S.units_ready, 0, err, ab, lim);
            if (small) {
                wait_phase(base + kPhFinQ);
            } else {
                // ------------------------------------------------ q, k, v of this CTA's attention units
                // The QKV partials summed, times 1/rms; RoPE on q and k; q pre-scaled by log2(e)/sqrt(hd)
                // for the exp2 softmax; fp16.  Splits of a row on several CTAs sum the same partials (and
                // store the same values): cheaper than a phase of its own, with an arrival and a wait.
                // 1.5B kernel, ms as a phase of its own -> here: 16 rows of 60 positions 1.145 -> 1.112, 26 rows
                // 1.202 -> 1.155, 64 rows 1.526 -> 1.445, 128 rows of 500 2.378 -> 2.273; 16 rows of 2000
                // positions, eight splits each, 1.355 -> 1.328.  (With a warp per group, whose halves
                // split the contributors: 80 rows 1.782 -> 1.800, 3B 26 rows 1.950 -> 1.989.)
                // A half warp takes a group of 64 weight rows; a head's weight rows come in 16s, 8 dims and
                // their rotation partners, so lane % 16 holds 4 dims and lane ^ 2 their partners.
                wait_phase(base + kPhQKV);
                const int half_hd = hd >> 1;
                int w = 2 * cw;  // this warp's next two groups, counted from the current unit's first
#pragma unroll 1
                for (int i = 0; i < n; ++i) {
                    const AttUnit &u = cta_unit(p, S, a0, i, 0);
                    const int r = u.row;
                    if (i >= p.KVH && cta_unit(p, S, a0, i - p.KVH, 1).row == r) continue;  // (an earlier split of the row)
                    // the groups that hold the unit's q heads, its k and its v
                    const int q0 = u.kvh * Gq * hd / 64, nq = ((u.kvh + 1) * Gq * hd + 63) / 64 - q0;
                    const int k0 = (p.H + u.kvh) * hd / 64, nk = ((p.H + u.kvh + 1) * hd + 63) / 64 - k0;
                    const int v0 = (p.H + p.KVH + u.kvh) * hd / 64, ng = nq + nk + ((p.H + p.KVH + u.kvh + 1) * hd + 63) / 64 - v0;
#pragma unroll 1
                    for (; w < ng; w += 16) {
                        const int y = min(w + (lane >> 4), ng - 1);  // (both halves the last one: the same values stored twice)
                        const int n0 = (y < nq ? q0 + y : y < nq + nk ? k0 + y - nq : v0 + y - nq - nk) * 64 + (lane & 15) * 4;
                        const int head = n0 / hd, j = n0 - head * hd;
                        const bool isq = head < p.H, isk = !isq && head < p.H + p.KVH, hi = (j & 8) != 0;
                        const int fr = (j >> 4) * 8 + (j & 7), d0 = hi ? fr + half_hd : fr;
                        // the row's sum-of-squares partials and rotation factors load with the QKV partials
                        const float sq = lane < d / 64 ? __ldcg(&p.ssqA[lane * p.rows_cap + r]) : 0.f;
                        const int pos = S.rowpos[r];
                        float4 c0 = make_float4(1.f, 0.f, 1.f, 0.f), c1 = c0;  // (cos, sin) of two dims each
                        if (isq || isk) {
                            const float4 *rp = reinterpret_cast<const float4 *>(p.rope + (int64_t)pos * half_hd + fr);
                            c0 = __ldg(rp);
                            c1 = __ldg(rp + 1);
                        }
                        const int t = n0 / kTileN;
                        const float4 x = part_sum(contributors(kGQKV, t), t, r * kTileN + n0 - t * kTileN, false);
                        const float rs = rsqrtf(warp_sum(sq) / (float)d + p.eps) * (isq ? p.scale_log2 : 1.f);
                        float4 o;
                        o.x = __shfl_xor_sync(0xffffffffu, x.x, 2);
                        o.y = __shfl_xor_sync(0xffffffffu, x.y, 2);
                        o.z = __shfl_xor_sync(0xffffffffu, x.z, 2);
                        o.w = __shfl_xor_sync(0xffffffffu, x.w, 2);
                        const float sg = hi ? 1.f : -1.f;  // rotate the pairs (i, i + hd/2); identity for v
                        const uint16_t h[4] = {f32_to_f16_sat((x.x * c0.x + sg * (o.x * c0.y)) * rs),
                                               f32_to_f16_sat((x.y * c0.z + sg * (o.y * c0.w)) * rs),
                                               f32_to_f16_sat((x.z * c1.x + sg * (o.z * c1.y)) * rs),
                                               f32_to_f16_sat((x.w * c1.z + sg * (o.w * c1.w)) * rs)};
                        *reinterpret_cast<uint2 *>(p.qkv16 + r * p.nqkv + head * hd + d0) = pack4(h);
                    }
                    w -= (ng + 1) & ~1;
                }
                named_bar_sync(1, kMegaCThreads);
                if (ctid == 0) atomicAdd(&p.cnt[(base + kPhFinQ) * kCntStride], 1ull);  // (few rows count on it)
            }
            // -------------------------------------------------------- attention
            // units alternate between the two warp groups: group h (warps 3..6 / 7..10, named
            // barrier 2 + h) runs the units (gi + i) & 1 == h.  Each warp of a group takes 32 positions
            // of every KV block by itself -- scores, probabilities and output sum stay in its registers
            // (online softmax, warp-level MMAs; the probabilities turn from accumulator into operand
            // by an 8 x 8 transpose), and nothing waits for another warp until the unit's end, where
            // the four warps' states are joined in shared memory.
            // Bound by the chain of a unit: phase wait, q, its blocks (about 1.1 us each once the two
            // that the ring prefetches are used up), join, split merge.  With 32 positions per warp for the
            // scores but 32 dims per warp for the output, as before, P went through shared memory behind
            // two barriers a block; and the ring's prefetch stopped at the block with the new
            // position until the phase that wrote it there was over.  1.5B kernel, ms before -> after:
            // 16 rows of 800 positions 1.337 -> 1.320, 64 of 600 1.791 -> 1.765, 128 of 300
            // 2.310 -> 2.280, one row of 384 1.145 -> 1.152 (its join costs more than the barriers did).
            const int hb = 2 + half;     // this group's named barrier
            const int ht = ctid & 127;   // thread index within the group
            const int hq = ht >> 5;      // warp within the group
            // ring entries of the phase's KV blocks: per unit pair, block by block, the K of
            // the pair's units, then their V^T (the W producer's order)
            uint32_t wpair = wring;
            const int g8 = lane >> 2, t4 = lane & 3;     // mma fragment row (head) / column pair
            const int kst = hd >> 4;                      // k-steps of q.k (16 dims each)
            float *mo = reinterpret_cast<float *>(sX) + half * 4 * 8 * kAttORow;  // [warp][head][dim], X stages' room
            // a tile's slot goes back to the producer once the group's four warps have read it
            auto kv_release = [&](uint32_t e) {
                __syncwarp();
                if (lane == 0 && atom_add_acq_rel_cta(&S.kvrel[wslot(e)], 1) == 3) {
                    S.kvrel[wslot(e)] = 0;
                    mbar_arrive(&S.wempty[wslot(e)]);
                }
            };
#pragma unroll 1
            for (int ip = 0; ip < n; ip += 2) {
                const bool two = ip + 1 < n;
                const int x = ((gi + ip) & 1) == half ? 0 : 1;  // our unit of the pair
                const AttUnit &u = cta_unit(p, S, a0, ip + (two ? x : 0), 0);
                const int nbo = two ? cta_unit(p, S, a0, ip + (x ^ 1), 1).nb : 0;  // the other unit's blocks
                const uint32_t w0 = wpair;
                wpair += 2u * (uint32_t)(u.nb + nbo);
                if (x == 1 && !two) continue;
                const int jm = min(u.nb, nbo);
                auto ent = [&](int j, int kv) -> uint32_t {
                    return j < jm ? w0 + 4u * j + 2u * kv + x : w0 + 4u * jm + 2u * (j - jm) + kv;
                };
                // ---- q of the unit's heads as mma B fragments (q^T: k = dim, n = head g8)
                uint32_t qf[8][2];
                {
                    const bool hv = g8 < Gq;
                    const uint16_t *qh = p.qkv16 + u.row * p.nqkv + (u.kvh * Gq + (hv ? g8 : 0)) * hd + 2 * t4;
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {
                        const bool ok = hv && ks < kst;
                        qf[ks][0] = ok ? __ldcg(reinterpret_cast<const unsigned int *>(qh + 16 * ks)) : 0u;
                        qf[ks][1] = ok ? __ldcg(reinterpret_cast<const unsigned int *>(qh + 16 * ks + 8)) : 0u;
                    }
                }
                // ---- the new position's k and v, if it is one of this warp's: four dims a lane
                const int pp = (u.ctx - 1) % kKVPos;
                const bool mine_new = u.last && (pp >> 5) == hq && 4 * lane < hd;
                uint2 kn = make_uint2(0, 0), vn = kn;
                uint8_t *blkn = nullptr;
                if (mine_new) {
                    blkn = kv_addr(p, l, S.rowblk[u.row], u.kvh);
                    const uint16_t *src = p.qkv16 + u.row * p.nqkv + (p.H + u.kvh) * hd + 4 * lane;
                    kn = __ldcg(reinterpret_cast<const uint2 *>(src));
                    vn = __ldcg(reinterpret_cast<const uint2 *>(src + p.KVH * hd));
                }
                // ---- per block: S^T = K q^T over this warp's 32 positions, probabilities against the
                // running max, which is re-based only when a score exceeds it by more than the headroom;
                // O^T += V^T P^T.  Thread (g8, t4): positions 16 i + g8 + {0, 8}, heads 2 t4 + {0, 1}; dims
                // 16 i + g8 + {0, 8} of the output.
                float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f}, o[8][4];
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int q = 0; q < 4; ++q) o[i][q] = 0.f;
#pragma unroll 1
                for (int jb = 0; jb < u.nb; ++jb) {
                    const int nj = min(kKVPos, u.n - jb * kKVPos) - 32 * hq;  // this warp's positions: below nj
                    const uint32_t ek = ent(jb, 0), ev = ent(jb, 1);
                    const bool add_new = mine_new && jb == u.nb - 1;
                    kv_wait(ek);
                    if (add_new) {  // into the tile that only this warp reads there, and into the cache
                        *reinterpret_cast<uint2 *>(sW + (size_t)wslot(ek) * kSlotBytes + kv_k_off(pp, 4 * lane)) = kn;
                        *reinterpret_cast<uint2 *>(blkn + kv_k_off(pp, 4 * lane)) = kn;
                        fence_proxy_async_smem();
                    }
                    __syncwarp();
                    uint32_t pf[2][2];  // P^T of 16 positions each as mma B fragments
                    if (nj > 0) {
                        const int pr = 32 * hq + (lane & 15);
                        const uint32_t krow = smem_u32(sW) + wslot(ek) * kSlotBytes + pr * 128;
                        float sc[2][4];
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int q = 0; q < 4; ++q) sc[i][q] = 0.f;
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks) {
                            if (ks < kst) {
                                const uint32_t off = (ks >> 2) * 16384 + ((((2 * ks & 7) + (lane >> 4)) ^ (pr & 7)) << 4);
#pragma unroll
                                for (int i = 0; i < 2; ++i) {
                                    uint32_t a[4];
                                    ldsm_x4(krow + off + i * 2048, a);
                                    mma_f16_16816(sc[i], a, qf[ks][0], qf[ks][1]);
                                }
                            }
                        }
                        float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                if (16 * i + g8 + 8 * (q >> 1) >= nj) sc[i][q] = -INFINITY;
                                mx[q & 1] = fmaxf(mx[q & 1], sc[i][q]);
                            }
#pragma unroll
                        for (int q = 0; q < 2; ++q)
#pragma unroll
                            for (int x2 = 4; x2 < 32; x2 <<= 1) mx[q] = fmaxf(mx[q], __shfl_xor_sync(0xffffffffu, mx[q], x2));
                        // (always on the first block)
                        if (__any_sync(0xffffffffu, mx[0] - m[0] > S.p_headroom || mx[1] - m[1] > S.p_headroom)) {
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const float mnew = fmaxf(m[q], mx[q]), alpha = exp2f(m[q] - mnew);
                                m[q] = mnew;
                                l[q] *= alpha;
#pragma unroll
                                for (int i = 0; i < 8; ++i) {
                                    o[i][q] *= alpha;
                                    o[i][q + 2] *= alpha;
                                }
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int y = 0; y < 2; ++y) {  // positions 16 i + 8 y ..
                                const float p0 = exp2f(sc[i][2 * y] - m[0]), p1 = exp2f(sc[i][2 * y + 1] - m[1]);
                                l[0] += p0;
                                l[1] += p1;
                                pf[i][y] = movmatrix_trans((uint32_t)f32_to_f16_sat(p0) | ((uint32_t)f32_to_f16_sat(p1) << 16));
                            }
                    }
                    kv_release(ek);
                    kv_wait(ev);
                    if (add_new) {
                        uint8_t *tile = sW + (size_t)wslot(ev) * kSlotBytes - 32768;
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const uint16_t v = (uint16_t)((e < 2 ? vn.x : vn.y) >> (16 * (e & 1)));
                            const int off = kv_v_off(pp, 4 * lane + e);
                            *reinterpret_cast<uint16_t *>(tile + off) = v;
                            *reinterpret_cast<uint16_t *>(blkn + off) = v;
                        }
                        fence_proxy_async_smem();
                    }
                    __syncwarp();
                    if (nj > 0) {
                        const int dr = lane & 15;
                        const uint32_t vrow = smem_u32(sW) + wslot(ev) * kSlotBytes + (hq >> 1) * 16384 + dr * 128;
#pragma unroll
                        for (int kk = 0; kk < 2; ++kk) {  // positions 16 kk .. of the warp's
                            const uint32_t off = ((uint32_t)((hq & 1) * 4 + 2 * kk + (lane >> 4)) ^ (dr & 7)) << 4;
#pragma unroll
                            for (int i = 0; i < 8; ++i)  // dims 16 i ..
                                if (16 * i < hd) {
                                    uint32_t a[4];
                                    ldsm_x4(vrow + off + i * 2048, a);
                                    mma_f16_16816(o[i], a, pf[kk][0], pf[kk][1]);
                                }
                        }
                    }
                    kv_release(ev);
                }
                // ---- the four warps' states: weights 2^(m_w - M), sums in warp order
#pragma unroll
                for (int q = 0; q < 2; ++q) {
#pragma unroll
                    for (int x2 = 4; x2 < 32; x2 <<= 1) l[q] += __shfl_xor_sync(0xffffffffu, l[q], x2);
                    if (g8 == 0) S.red[half][hq][2 * t4 + q] = m[q];
                }
                named_bar_sync(hb, 128);
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int h = 2 * t4 + q;
                    const float M = fmaxf(fmaxf(S.red[half][0][h], S.red[half][1][h]),
                                          fmaxf(S.red[half][2][h], S.red[half][3][h]));
                    const float w = exp2f(m[q] - M);  // 0 for a warp without positions
                    if (g8 == 0) S.red2[half][hq][h] = l[q] * w;
                    float *dst = mo + (hq * 8 + h) * kAttORow + g8;
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (16 * i < hd) {
                            dst[16 * i] = o[i][q] * w;
                            dst[16 * i + 8] = o[i][q + 2] * w;
                        }
                }
                named_bar_sync(hb, 128);
                // ---- output (single split) or partial + split merge; thread ht: dim ht of every head
                const bool single = u.nsplit == 1;
                const int dd = ht;
                float *mine = p.part + ((int64_t)u.item * p.KVH + u.kvh) * Gq * (hd + 2);
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    if (g < Gq && dd < hd) {
                        float v = 0.f, L = 0.f;
#pragma unroll
                        for (int w = 0; w < 4; ++w) v += mo[(w * 8 + g) * kAttORow + dd];
                        if (single) {
#pragma unroll
                            for (int w = 0; w < 4; ++w) L += S.red2[half][w][g];
                            uint16_t hv, lv;
                            split_bf16(v / L, hv, lv);
                            uint8_t *dst = p.att + att_off(u.row, (u.kvh * Gq + g) * hd + dd);
                            *reinterpret_cast<uint16_t *>(dst) = hv;
                            *reinterpret_cast<uint16_t *>(dst + lo_off) = lv;
                        } else {
                            mine[g * (hd + 2) + 2 + dd] = v;
                        }
                    }
                }
                if (single) {
                    named_bar_sync(hb, 128);  // the states' room is free again
                    continue;
                }
                if (dd < Gq) {
                    float M = S.red[half][0][dd], L = S.red2[half][0][dd];
#pragma unroll
                    for (int w = 1; w < 4; ++w) {
                        M = fmaxf(M, S.red[half][w][dd]);
                        L += S.red2[half][w][dd];
                    }
                    mine[dd * (hd + 2)] = M;
                    mine[dd * (hd + 2) + 1] = L;
                }
                named_bar_sync(hb, 128);
                if (ht == 0) {  // one acquire-release count: publishes this split, sees the others
                    const int old = atom_add_acq_rel_gpu(&p.att_cnt[u.row * p.KVH + u.kvh], 1);
                    S.last_flag2[half] = old == u.nsplit - 1;
                    if (S.last_flag2[half]) p.att_cnt[u.row * p.KVH + u.kvh] = 0;
                }
                named_bar_sync(hb, 128);
                if (S.last_flag2[half]) {  // merge the row's splits in split order
                    const int ns = min(u.nsplit, kMegaMaxSplits);
                    const int sp_stride = p.KVH * Gq * (hd + 2), hs = hd + 2;
                    const float *pb = p.part + ((int64_t)__ldg(&p.c.row_item0[u.row]) * p.KVH + u.kvh) * Gq * hs;
                    float acc[8];
#pragma unroll
                    for (int g = 0; g < 8; ++g) acc[g] = 0.f;
#pragma unroll 1
                    for (int s0 = 0; s0 < ns; s0 += 2) {
                        // two splits' outputs in flight (thread dd: dim dd of every head; more would spill
                        // registers); the first two load together with the split weights' inputs
                        const float *src = pb + s0 * sp_stride + 2 + dd;
                        float v[2][8];
#pragma unroll
                        for (int q = 0; q < 2; ++q, src += sp_stride)
#pragma unroll
                            for (int g = 0; g < 8; ++g)
                                v[q][g] = (dd < hd && g < Gq && s0 + q < ns) ? __ldcg(src + g * hs) : 0.f;
                        if (s0 == 0) {
                            // split weights 2^(m_s - M), total weight L per head (warp hq: heads hq, hq + 4)
#pragma unroll 1
                            for (int g = hq; g < Gq; g += 4) {
                                float ms[3], ls[3];
                                float Mx = -INFINITY;
#pragma unroll
                                for (int q = 0; q < 3; ++q) {
                                    const int sp = lane + 32 * q;
                                    ms[q] = sp < ns ? __ldcg(pb + sp * sp_stride + g * hs) : -INFINITY;
                                    ls[q] = sp < ns ? __ldcg(pb + sp * sp_stride + g * hs + 1) : 0.f;
                                    Mx = fmaxf(Mx, ms[q]);
                                }
#pragma unroll
                                for (int o2 = 16; o2 > 0; o2 >>= 1) Mx = fmaxf(Mx, __shfl_xor_sync(0xffffffffu, Mx, o2));
                                float L = 0.f;
#pragma unroll
                                for (int q = 0; q < 3; ++q) {
                                    const int sp = lane + 32 * q;
                                    const float w = sp < ns ? exp2f(ms[q] - Mx) : 0.f;
                                    if (sp < ns) S.mw[half][g][sp] = w;
                                    L += w * ls[q];
                                }
                                L = warp_sum(L);
                                if (lane == 0) S.ml[half][g] = L;
                            }
                            named_bar_sync(hb, 128);
                        }
#pragma unroll
                        for (int q = 0; q < 2; ++q)
#pragma unroll
                            for (int g = 0; g < 8; ++g)
                                if (g < Gq && s0 + q < ns) acc[g] += S.mw[half][g][s0 + q] * v[q][g];
                    }
                    if (dd < hd) {
#pragma unroll
                        for (int g = 0; g < 8; ++g)
                            if (g < Gq) {
                                uint16_t hv, lv;
                                split_bf16(acc[g] / S.ml[half][g], hv, lv);
                                uint8_t *dst = p.att + att_off(u.row, (u.kvh * Gq + g) * hd + dd);
                                *reinterpret_cast<uint16_t *>(dst) = hv;
                                *reinterpret_cast<uint16_t *>(dst + lo_off) = lv;
                            }
                    }
                }
                named_bar_sync(hb, 128);
            }
            wring = wpair;
            gi += n;
            fence_proxy_async_smem();  // (the X stages are targets of bulk copies again)
            arrive(base + kPhAtt, true);
        }
        if (small && k != 2) {
            // ------------------------------------------------ column-owned q/k/v or O projection
            // Each CTA's few features hold the whole K, so what follows the sums is applied at
            // once.  Thread: feature c = ctid % 16 of its (unit, row) elements.
            //   q/k/v: RMSNorm scale, RoPE (a unit is 8 dims of a head and their rotation
            //     partners), fp16.
            //   O: x += sum, the MLP norm's input, sums of squares (one partial per 16 features).
            wait_phase(k == 0 ? base - 1 : base + kPhAtt);
            const GemmPlan &g = S.plan[k];
            const uint8_t *X = k == 0 ? p.xg : p.att;
            float *red = reinterpret_cast<float *>(sX);  // no copy targets the X stages during these phases
            const int half_hd = hd >> 1, c = ctid & 15, r = (ctid >> 4) & 7, m = ctid >> 7;
            SegWalk walk(g);
            Seg sg;
#pragma unroll 1
            while (walk.next(g, sg)) {
                const bool live = r < R && m * kOwnCols < sg.n;  // this thread's element (unit m, feature c, row r)
                const int n0 = sg.col0 + m * kOwnCols, head = n0 / hd;
                const bool rot = head < p.H + p.KVH;
                float2 pre = make_float2(1.f, 0.f);  // (cos, sin) or (residual, norm weight), in flight with the operand
                if (live) {
                    if (k != 0) {
                        pre.x = __ldcg(p.x + r * d + n0 + c);
                        pre.y = bf16_to_f32(__ldg(p.mlp_norm + l * d + n0 + c));
                    } else if (rot) {
                        pre = __ldg(&p.rope[S.rowpos[r] * half_hd + (n0 - head * hd) / 2 + (c & 7)]);
                    }
                }
                if (k == 0) load_rstd(p.ssqA, d / 64);
                small_k(S, sW, red, X, R16c, g.kch, sg, wring, cw, lane, kv_wait, nws_mul);
                named_bar_sync(1, kMegaCThreads);
                const int E = sg.entries();
                if (ctid == 0)  // the slots not yet returned
                    for (int e = (E - 1) / S.nws * S.nws; e < E; ++e) mbar_arrive(&S.wempty[wslot(wring + e)]);
                wring += (uint32_t)E;
                float v = 0.f;
                if (live) {
#pragma unroll
                    for (int w = 0; w < 8; ++w) v += red[((w * kSmallUnits + m) * kOwnCols + c) * 8 + ((r + c) & 7)];
                }
                uint32_t w0, w1;  // what this lane keeps and what its neighbour lane ^ 1 takes
                float sq = 0.f;
                if (k == 0) {
                    const float vp = __shfl_xor_sync(0xffffffffu, v, 8);
                    const float y = v * pre.x + (c < 8 ? -1.f : 1.f) * (vp * pre.y);
                    w0 = w1 = f32_to_f16_sat(y * ((live ? S.rstd[r] : 0.f) * (head < p.H ? p.scale_log2 : 1.f)));
                } else {
                    const float x = pre.x + v;
                    if (live) p.x[r * d + n0 + c] = x;
                    uint16_t h, lo;
                    split_bf16(x * pre.y, h, lo);
                    w0 = (c & 1) ? lo : h;  // even lanes store both hi parts, odd lanes both lo parts
                    w1 = (c & 1) ? h : lo;
                    sq = live ? x * x : 0.f;
#pragma unroll
                    for (int o = 1; o < 16; o <<= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
                }
                const uint32_t wn = __shfl_xor_sync(0xffffffffu, w1, 1);
                const uint32_t pk = (c & 1) ? wn | (w0 << 16) : w0 | (wn << 16);  // features c & ~1, c | 1
                if (live && k == 0) {
                    const int dim = (n0 - head * hd) / 2 + (c & 7) + (c < 8 ? 0 : half_hd);
                    if ((c & 1) == 0) *reinterpret_cast<uint32_t *>(p.qkv16 + r * p.nqkv + head * hd + dim) = pk;
                } else if (live) {
                    *reinterpret_cast<uint32_t *>(p.xg + xblk_off(r, (n0 + c) & ~1, R16c) + ((c & 1) ? kLoOff : 0)) = pk;
                    if (c == 0) p.ssqM[n0 / kOwnCols * p.rows_cap + r] = sq;
                }
                named_bar_sync(1, kMegaCThreads);  // red is free again
            }
            fence_proxy_async_smem();  // (its room is a target of bulk copies again)
            arrive(base + (k == 0 ? kPhFinQ : kPhFinO), k == 1);
            // (the split-K phase's counter keeps step: a later launch with more rows waits on it)
            if (ctid == 0) atomicAdd(&p.cnt[(base + (k == 0 ? kPhQKV : kPhO)) * kCntStride], 1ull);
        } else {
        // ---------------------------------------------------------------- split-K GEMM
        // this CTA's partial tiles: row my_row, columns [128 half, +128) of the tile
        {
            const GemmPlan &g = S.plan[k];
            SegWalk walk(g);
            Seg sg;
#pragma unroll 1
            while (walk.next(g, sg)) {
                wring += (uint32_t)sg.entries();
                const uint32_t a = acc_wait();
                if (quarter_live && half * 128 < sg.n) {
                    float *dst = p.gpart + ((cta + sg.t) * p.rows_cap + (act ? my_row : 0)) * kTileN + half * 128;
#pragma unroll 1
                    for (int cc = 0; cc < 4; ++cc) {
                        float v[32];
                        tmem_ld_32x32b_x32(tmem + lane_base + a * kTileN + half * 128 + cc * 32, v);
                        float w[16];
                        pair_part(v, w);
#pragma unroll 1
                        for (int q = second ? 1 : 0; q < (pair && !second ? 1 : 2); ++q) {  // 16 columns each
                            if (!act) continue;
                            float *o = dst + cc * 32 + q * 16;
#pragma unroll
                            for (int e = 0; e < 16; ++e) w[e] += q ? v[16 + e] : v[e];
                            st_global_v8(o, w);
                            st_global_v8(o + 8, w + 8);
                            if (!pair) {
#pragma unroll
                                for (int e = 0; e < 16; ++e) w[e] = 0.f;
                            }
                        }
                    }
                }
                acc_release(a);
            }
            arrive(base + (k == 0 ? kPhQKV : k == 1 ? kPhO : kPhDown), false);
        }
        }
        if (++k == 3) {
            k = 0;
            ++l;
        }
    }

    // ---------------------------------------------------------------- lm_head + Gumbel-max
    // logits = (x_g W_lm^T) / rms(x) for the live rows, fused with the temperature-1 sampler:
    // each thread scans its columns of the CTA's in increasing token order, adds the
    // Gumbel noise g(row key, token) and keeps the first maximum of logit + g; the per (row,
    // CTA, half) maxima go to the bookkeeping kernel, which takes the row's argmax (ties to
    // the lowest token id).  Products and sums are rounded separately (no contraction), as
    // the sampler on stored logits would do them.  The logits themselves are written only
    // when requested (teacher forcing).
    // (Each lane finishes its columns one after the other, so a small vocabulary in whole 256-token tiles
    // on two CTAs took 12 us of 54: it is shared in 16-token units over all CTAs.  Vocabulary of 512
    // and 2 rows, kernel: 51.1 -> 45.7 us; 25 rows: 66.4 -> 61.1.)
    wait_phase(kPhasesPerLayer * p.layers);
    load_rstd(p.ssqA, d / 64);
    named_bar_sync(1, kMegaCThreads);
    const GemmPlan &g = S.plan[kGLM];
    const float rs = act ? S.rstd[my_row] : 0.f;
    const uint64_t seed = act ? __ldg(&p.c.row_seed[my_row]) : 0ull;
    float best = -INFINITY;  // running over this thread's tiles (its row and columns)
    int bi = 0x7fffffff;
    SegWalk walk(g);
    Seg sg;
#pragma unroll 1
    while (walk.next(g, sg)) {
        const uint32_t a = acc_wait();
        const int hc = 32 * ((sg.n + 63) / 64);  // a half's columns: from half * hc on
        if (quarter_live) {
#pragma unroll 1
            for (int c0 = half * hc; c0 < min(sg.n, half * hc + hc); c0 += 32) {
                float v[32];
                tmem_ld_32x32b_x32(tmem + lane_base + a * kTileN + c0, v);
                float w[16];
                pair_part(v, w);
                // 16 columns at a time; each lane of a pair takes one half of the 32
#pragma unroll 1
                for (int q = second ? 1 : 0; q < (pair && !second ? 1 : 2); ++q) {
                    if (!act || c0 + q * 16 >= sg.n) continue;
                    float z[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) z[e] = __fmul_rn((q ? v[16 + e] : v[e]) + w[e], rs);
                    const int nb = sg.col0 + c0 + q * 16;
                    if (p.write_logits) {
                        float4 *o = reinterpret_cast<float4 *>(p.logits + (int64_t)my_row * p.V + nb);
#pragma unroll
                        for (int e = 0; e < 4; ++e) o[e] = make_float4(z[4 * e], z[4 * e + 1], z[4 * e + 2], z[4 * e + 3]);
                    }
                    // Only tokens whose noise could lift them to the best so far are evaluated
                    // exactly (noise_cut).  `best` runs over all of this thread's columns; before the
                    // first maximum, the sum of the token of the largest noise stands in for it.
                    float low = best;
                    if (best == -INFINITY) {
                        uint32_t most = 0;
                        int me = 0;
#pragma unroll 1
                        for (int e = 0; e < 16; ++e) {
                            const uint32_t code = (uint32_t)(splitmix_at(seed, (uint64_t)(nb + e) + 1) >> 40);
                            if (code > most) { most = code; me = e; }
                        }
                        float ze = z[0];
#pragma unroll
                        for (int i = 1; i < 16; ++i) ze = (i == me) ? z[i] : ze;
                        low = __fadd_rn(ze, gumbel_from_hash(splitmix_at(seed, (uint64_t)(nb + me) + 1)));
                    }
                    float vmax = z[0];
#pragma unroll
                    for (int e = 1; e < 16; ++e) vmax = fmaxf(vmax, z[e]);
                    const uint32_t thr = noise_cut(low, vmax);
                    uint32_t cand = 0;
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        cand |= (uint32_t)((uint32_t)(splitmix_at(seed, (uint64_t)(nb + e) + 1) >> 40) >= thr) << e;
#pragma unroll 1
                    while (cand) {  // candidates in increasing token order: the first maximum is kept
                        const int e = __ffs(cand) - 1;
                        cand &= cand - 1;
                        float ze = z[0];
#pragma unroll
                        for (int i = 1; i < 16; ++i) ze = (i == e) ? z[i] : ze;
                        const float zg = __fadd_rn(ze, gumbel_from_hash(splitmix_at(seed, (uint64_t)(nb + e) + 1)));
                        if (zg > best) { best = zg; bi = nb + e; }
                    }
                }
            }
        }
        acc_release(a);
    }
    // this (CTA, half)'s maximum (-inf where it has no columns); the lanes of a pair hold disjoint
    // columns (ties to the lower id)
    if (pair) {
        const float ov = __shfl_xor_sync(0xffffffffu, best, 8);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, 8);
        if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
    }
    if (act && !second) {
        p.c.arg_val[(my_row * G + cta) * 2 + half] = best;
        p.c.arg_idx[(my_row * G + cta) * 2 + half] = bi;
    }
    named_bar_sync(1, kMegaCThreads);
    if (ctid == 0) MEGA_STAMP(1 + kPhasesPerLayer * p.layers, 0);
}

// ------------------------------------------------------------------------------ kernel
__global__ void __launch_bounds__(kMegaThreads, 1) decode_step_kernel(const __grid_constant__ MegaParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *sW = base;
    MegaSmem &S = *reinterpret_cast<MegaSmem *>(sW + kRingBytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    StepVars *V = p.c.v;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxWSlots; ++s) {
            mbar_init(&S.wfull[s], 1);
            mbar_init(&S.wempty[s], 1);
            mbar_init(&S.kvready[0][s], 1);
            mbar_init(&S.kvready[1][s], 1);
            S.kvrel[s] = 0;
        }
        for (int s = 0; s < kMaxXStages; ++s) { mbar_init(&S.xfull[s], 1); mbar_init(&S.xempty[s], 1); }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&S.acc_full[a], 1);
            mbar_init(&S.acc_empty[a], 8);
        }
        mbar_init(&S.drain, 1);
        mbar_init(&S.units_ready, 1);
        const int live = *(volatile int *)&V->live;
        const int rows = max(0, min(live, p.rows_cap));
        S.rows = rows;
        S.rows16 = max(16, (rows + 15) & ~15);
        S.small = live <= kSmallRows;
        // X stages of several k-chunks each where the rows are few (fewer waits and commits per MMA), as
        // many as fit after the W slots
        S.nws = ring_slots(rows);
        S.xchunk = x_chunk_bytes(rows);
        S.xgroup = x_stage_chunks(rows);
        S.nx = x_stages(rows);
        S.n_items = *(volatile int *)&V->att_items;
        S.att_span = max(1, *(volatile int *)&V->att_span);
        S.target = (*(volatile unsigned long long *)p.epoch + 1ull) * gridDim.x;
        // failure limits of this call (sara_set_limits): read at run time, not baked into the graph
        const int64_t wl = p.c.kc->wait_ns;
        S.wait_ns = wl > 0 ? (uint64_t)wl : kWaitLimitNs;
        S.stall_idx = p.c.kc->stall_plus1 - 1;
        // phases that finalise their own sums count on the second of their two counters
        if (S.stall_idx > 0) {
            const int ph = (S.stall_idx - 1) % kPhasesPerLayer;
            if (ph == kPhGU - 1 || (S.small && (ph == kPhQKV || ph == kPhO))) ++S.stall_idx;
            if (ph == kPhFinQ && !S.small) --S.stall_idx;  // (the attention units' sums wait on the projection)
        }
        S.p_headroom = p.c.kc->eager_softmax ? 0.f : kSoftmaxHeadroom;
        S.abort = (*(volatile int *)&V->err & ERR_WAIT_TIMEOUT) != 0;
        fence_mbar_init();
    }
    if (threadIdx.x == 0) MEGA_STAMP(p.n_stamp_ph - 1, 0);  // kernel start
    const uint64_t t_start = globaltimer_ns();
    const bool small = *(volatile int *)&V->live <= kSmallRows;
    // the launch's GEMM shares and the contributors of the split-K tiles
    if (threadIdx.x >= 32 * 3 && threadIdx.x < 32 * 3 + 5)
        make_plan(p, S.plan[threadIdx.x - 96], threadIdx.x - 96, blockIdx.x, gridDim.x, small);
    if (threadIdx.x >= 128 && threadIdx.x < 128 + 3 * kPlanTiles) {
        const int which = (threadIdx.x - 128) / kPlanTiles, t = (threadIdx.x - 128) % kPlanTiles;
        GemmPlan g;
        make_plan(p, g, which, 0, gridDim.x, false);
        if (t < (g.N + kTileN - 1) / kTileN) S.tile_cta[which][t] = tile_ctas(p, g, which, t, gridDim.x);
    }
    if (warp == 1) {
        tmem_alloc(&S.tmem_base, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_base;
    uint8_t *sX = sW + (size_t)S.nws * kSlotBytes;
    const bool run = !S.abort && S.rows > 0;
    if (run) {
        if (warp == 0) {
            fill_att_blocks(p, S, lane);
            if (lane == 0) mbar_arrive(&S.units_ready);
            mega_w_producer(p, S, sW);
        } else if (warp == 1) {
            mega_mma(p, S, sW, sX, tmem);
        } else if (warp == 2) {
            mega_x_producer(p, S, sX);
        } else {
            mega_compute(p, S, sW, sX, tmem);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, kTmemCols);
    // every CTA read the epoch before any CTA could pass the first phase; the last phase's
    // wait in CTA 0 therefore happens after all reads
    if (run && threadIdx.x == 0 && blockIdx.x == 0) atomicAdd(p.epoch, 1ull);
    // launch duration for the step's kernel-time total (the bookkeeping kernel folds it in)
    if (run && threadIdx.x == 0 && p.ktime) {
        atomicMin(&p.ktime[0], (unsigned long long)t_start);
        atomicMax(&p.ktime[1], (unsigned long long)globaltimer_ns());
    }
}

// ------------------------------------------------------------------------------ layout kernels
// Rows of a source matrix in the blocked matrix that it is a part of.
enum : int {
    kRowsPlain = 0,  // row + row0
    kRowsHead = 1,   // q, k, v: each head's rows in qkv_row order, + row0
    kRowsAlt = 2,    // gate, up: alternate blocks of 8 rows (row0 = 0: gate, 8: up)
};
// Row-major W [n_src][K] (bf16, 16-byte aligned) into chunk-major blocks of a matrix of N rows:
// k-chunk kc holds its 64 columns of every row (128 bytes a row), 16-byte granule j of row r stored
// at granule j ^ (r % 8), so any run of rows of a chunk that starts at a multiple of 8 is one
// contiguous piece.  K must be a multiple of 64.
static __global__ void block_weights_kernel(const uint16_t *src, uint8_t *dst, int n_src, int K, int N, int rows, int row0,
                                            int head_dim) {
    const int gpr = K / 8;
    const int64_t total = (int64_t)n_src * gpr;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        int n = (int)(e / gpr);
        const int j = (int)(e - (int64_t)n * gpr);
        const uint4 v = *reinterpret_cast<const uint4 *>(src + (int64_t)n * K + (int64_t)j * 8);
        if (rows == kRowsHead) n = n / head_dim * head_dim + qkv_row(n % head_dim, head_dim / 2);
        else if (rows == kRowsAlt) n = (n >> 3) * 16 + (n & 7);
        n += row0;
        *reinterpret_cast<uint4 *>(dst + wblk_off(N, n, j >> 3) + (((j & 7) ^ (n & 7)) << 4)) = v;
    }
}

// KV set-up of the rollouts that join, from the prefill's row-major prompt KV ([2][n_kv][cap_p]
// [hd] per prompt slot and layer, positions < Lp - 1): (a) every fresh prompt's full blocks
// (positions < nsh * 128), which its rollouts share; (b) every new rollout's private block
// holding position Lp - 1 (slots new_slots[0 .. n_new)), filled with the prompt's tail positions
// nsh * 128 .. Lp - 2.  One thread per K granule (8 dims of a position) or V granule (8
// positions of a dim).
static __global__ void prompt_blocks_kernel(const uint16_t *pkv, uint8_t *kv, const StepPtrs c, int layers, int n_kv,
                                            int hd, int cap_p, int64_t kv_layer, int max_active) {
    pdl_wait_prior_grids();
    pdl_allow_dependents();
    const int n_new = c.v->n_new, n_fresh = c.v->n_fresh;
    const int Lp = c.kc->Lp, Lpre = Lp - 1;
    const int nsh = shared_blocks(Lp, kKVPos);
    const int gk = hd / 8;
    // per (layer, kv head) plane: K granules npos * gk, then V granules ceil(npos / 8) * hd
    const int na = nsh * kKVPos, nt = Lpre - na;  // positions of a shared plane / of a tail plane
    const int64_t per_a = (int64_t)na * gk + (int64_t)(na / 8) * hd;
    const int64_t per_b = (int64_t)nt * gk + (int64_t)((nt + 7) / 8) * hd;
    const int64_t tot_a = (int64_t)n_fresh * layers * n_kv * per_a;
    const int64_t total = tot_a + (int64_t)n_new * layers * n_kv * per_b;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        int64_t rem;
        int owner, npos, p0;  // owner: fresh prompt f or rollout slot s; positions [p0, p0 + npos)
        int64_t per;
        if (e < tot_a) {
            rem = e;
            per = per_a;
            npos = na;
            p0 = 0;
        } else {
            rem = e - tot_a;
            per = per_b;
            npos = nt;
            p0 = na;
        }
        const int64_t per_owner = (int64_t)layers * n_kv * per;
        owner = (int)(rem / per_owner);
        rem -= (int64_t)owner * per_owner;
        const int l = (int)(rem / ((int64_t)n_kv * per));
        rem -= (int64_t)l * n_kv * per;
        const int kvh = (int)(rem / per);
        rem -= (int64_t)kvh * per;
        const bool shared = e < tot_a;
        const int slot = shared ? 0 : c.new_slots[owner];
        const int ps = shared ? c.fresh_pslot[owner] : c.seq_pslot[slot];
        const uint16_t *kplane = pkv + (((int64_t)l * max_active + ps) * 2 * n_kv + kvh) * cap_p * hd;
        const uint16_t *vplane = kplane + (int64_t)n_kv * cap_p * hd;
        const int nk = npos * gk;
        int pos, dd = 0;
        bool isk = rem < nk;
        if (isk) {
            pos = p0 + (int)(rem / gk);
            dd = (int)(rem - (int64_t)(pos - p0) * gk) * 8;
        } else {
            rem -= nk;
            pos = p0 + (int)(rem / hd) * 8;
            dd = (int)(rem - (int64_t)((pos - p0) / 8) * hd);
        }
        const int b = pos / kKVPos;
        const int blk = shared ? ps * c.nsh_max + b : c.blk_tab[(int64_t)slot * c.nblk_max + b];
        uint8_t *dst = kv + l * kv_layer + ((int64_t)blk * n_kv + kvh) * kKVBlockBytes;
        if (isk) {
            const uint4 v = *reinterpret_cast<const uint4 *>(kplane + (int64_t)pos * hd + dd);
            *reinterpret_cast<uint4 *>(dst + kv_k_off(pos % kKVPos, dd)) = v;
        } else {
            uint32_t w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int pa = pos + 2 * q;
                const uint32_t x = pa < Lpre ? vplane[(int64_t)pa * hd + dd] : 0u;
                const uint32_t y = pa + 1 < Lpre ? vplane[(int64_t)(pa + 1) * hd + dd] : 0u;
                w[q] = x | (y << 16);
            }
            *reinterpret_cast<uint4 *>(dst + kv_v_off(pos % kKVPos, dd)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

}  // namespace sara
