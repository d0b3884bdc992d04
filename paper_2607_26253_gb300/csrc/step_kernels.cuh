// Small kernels of the step graph: embedding gather for the prefill rows (with the first
// RMSNorm's inputs), sampling reduction + per-step bookkeeping, and the teacher-forcing
// round setup.
#pragma once
#include "controller.cuh"
#include "device_common.cuh"
#include "step_state.cuh"

namespace sara {

// x_f32[r] = E[tok[r]]; xg[r] = x * g as a bf16 hi/lo pair; ssq[t][r] = sum over features
// [128t, 128t+128) of x^2.  One warp per row, four features a lane, so that a 128-feature sum is one
// warp reduction; bound by its stores (10 bytes a feature: 16,320 x 1,536 77 -> 42 us against a CTA
// per row with two barriers per 128 features).
static __global__ void __launch_bounds__(256) embed_kernel(const uint16_t *E, const uint16_t *g, const int *rows_dev,
                                                           const int *row_tok, int d, int rows_cap, int vocab,
                                                           float *x_f32, uint16_t *xg, uint16_t *xg_lo, float *ssq,
                                                           int *err) {
    pdl_wait_prior_grids();
    pdl_allow_dependents();
    const int rows = min(*rows_dev, rows_cap), lane = threadIdx.x & 31;
    for (int r = blockIdx.x * 8 + (threadIdx.x >> 5); r < rows; r += gridDim.x * 8) {
        int tok = row_tok[r];
        if (tok < 0 || tok >= vocab) {  // token ids come from the caller: never read outside E
            if (lane == 0) report_error(err, ERR_BOUNDS);
            tok = 0;
        }
        const uint16_t *er = E + (int64_t)tok * d;
#pragma unroll 4
        for (int t = 0; t < d / 128; ++t) {
            const int f = t * 128 + lane * 4;
            const uint2 e = __ldg(reinterpret_cast<const uint2 *>(er + f));
            const uint2 w = __ldg(reinterpret_cast<const uint2 *>(g + f));
            const float4 x = make_float4(bf16_to_f32(e.x & 0xffff), bf16_to_f32(e.x >> 16), bf16_to_f32(e.y & 0xffff),
                                         bf16_to_f32(e.y >> 16));
            uint16_t hi[4], lo[4];
            split_bf16(x.x * bf16_to_f32(w.x & 0xffff), hi[0], lo[0]);
            split_bf16(x.y * bf16_to_f32(w.x >> 16), hi[1], lo[1]);
            split_bf16(x.z * bf16_to_f32(w.y & 0xffff), hi[2], lo[2]);
            split_bf16(x.w * bf16_to_f32(w.y >> 16), hi[3], lo[3]);
            const int64_t o = (int64_t)r * d + f;
            *reinterpret_cast<float4 *>(x_f32 + o) = x;
            *reinterpret_cast<uint2 *>(xg + o) = pack4(hi);
            *reinterpret_cast<uint2 *>(xg_lo + o) = pack4(lo);
            const float s = warp_sum((x.x * x.x + x.y * x.y) + (x.z * x.z + x.w * x.w));
            if (lane == 0) ssq[(int64_t)t * rows_cap + r] = s;
        }
    }
}

// 256-thread exclusive scan helper (blockDim.x == 256): returns the prefix, sets total.
__device__ __forceinline__ int scan256(int v, int &total, int *warp_tot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    int before = 0, tot = 0;
    for (int w = 0; w < 8; ++w) {
        if (w < warp) before += warp_tot[w];
        tot += warp_tot[w];
    }
    __syncthreads();
    total = tot;
    return before + x - v;
}

// Sampling finish + step bookkeeping, after the decode-step kernel.  That kernel's lm_head
// epilogue left, per live row, the first maximum of logit + Gumbel noise of every (CTA, half of its
// columns) (arg_val / arg_idx [rows][lm_parts]); CTA r reduces row r's maxima
// to its token (ties: lowest token id).  The last CTA to finish appends each row's token to
// its rollout, retires rollouts that reached their length, compacts the live rows (order
// kept) and writes the next step's rows and attention items.
//
// use_more: the kernel ends a decode loop of the step graph and sets its condition: another step
// follows unless the controller has work (a round's last rollout finished, or on the asynchronous
// schedule a prompt's batch), an error was reported, or a bound is reached (the controller then
// reports it).
static __global__ void __launch_bounds__(256) sample_finish_kernel(StepPtrs c, cudaGraphConditionalHandle more,
                                                                   int use_more) {
    __shared__ int span_sm[kAttCands + 1];
    __shared__ float sv[8];
    __shared__ int si[8];
    __shared__ int s_last;
    __shared__ int warp_tot[8];
    pdl_wait_prior_grids();
    pdl_allow_dependents();
    StepVars &V = *c.v;
    const int live = V.live;
    const int r = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (r < live) {
        const int nparts = c.lm_parts;
        float best = -INFINITY;
        int bi = 0x7fffffff;
        for (int j = tid; j < nparts; j += blockDim.x) {
            const float v = __ldcg(&c.arg_val[(int64_t)r * nparts + j]);
            const int id = __ldcg(&c.arg_idx[(int64_t)r * nparts + j]);
            if (v > best || (v == best && id < bi)) { best = v; bi = id; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
        }
        if (lane == 0) { sv[warp] = best; si[warp] = bi; }
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < 8; ++w)
                if (sv[w] > best || (sv[w] == best && si[w] < bi)) { best = sv[w]; bi = si[w]; }
            c.sampled[r] = bi;
        }
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        const int old = atomicAdd(&V.fin_count, 1);
        s_last = (old == (int)gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid == 0) {
        V.fin_count = 0;
        // the preceding decode-step launch's duration into the step's kernel-time total
        if (V.kt1 > V.kt0) V.kernel_ns += (int64_t)(V.kt1 - V.kt0);
        V.kt0 = ~0ull;
        V.kt1 = 0ull;
    }
    if (live == 0) {
        if (use_more && tid == 0) cudaGraphSetConditional(more, 0u);
        return;
    }
    const StepConst &K = *c.kc;
    const int Lp = K.Lp, B = K.attn_chunk;
    const int nsh = shared_blocks(Lp, B);
    // bookkeeping over the live rows (several passes of 256)
    int out = 0;
    int top = V.blk_top, low = V.blk_low;  // the KV block free stack (same value in every thread)
    int stop = V.slot_top;                 // the free rollout slots (asynchronous schedule)
    for (int base = 0; base < live; base += 256) {
        const int i = base + tid;
        int keep = 0, slot = 0, gen = 0, next_tok = 0;
        if (i < live) {
            slot = c.row_slot[i];
            gen = c.seq_gen[slot];
            const int tok = __ldcg(&c.sampled[i]);
            if (K.teacher) {
                c.sampled_out[(int64_t)slot * K.T_forced + gen] = tok;
                next_tok = (gen + 1 < K.T_forced) ? c.forced[(int64_t)slot * K.T_forced + gen] : 0;
            } else {
                c.gen_tok[((int64_t)c.seq_q[slot] * K.k + c.seq_j[slot]) * K.max_gen + gen] = tok;
                next_tok = tok;
            }
            gen += 1;
            c.seq_gen[slot] = gen;
            keep = gen < c.seq_len[slot];
        }
        // KV blocks, in row order: a finished rollout returns its private blocks (positions
        // up to Lp - 2 + gen), then a kept one whose next position opens a block takes one
        int32_t *bt = c.blk_tab + (int64_t)slot * c.nblk_max;
        int nfree = 0, need = 0;
        if (i < live) {
            if (!keep) nfree = (Lp + gen - 2) / B - nsh + 1;
            else need = ((Lp - 1 + gen) % B) == 0;
        }
        int ftot;
        const int foff = scan256(nfree, ftot, warp_tot);
        for (int j = 0; j < nfree; ++j) c.blk_free[top + foff + j] = bt[nsh + j];
        top += ftot;
        __syncthreads();
        int atot;
        const int aoff = scan256(need, atot, warp_tot);
        if (need) {
            const int at = top - 1 - aoff;
            if (at >= 0) bt[(Lp - 1 + gen) / B] = c.blk_free[at];
            else report_error(&V.err, ERR_CAPACITY);
        }
        top = max(0, top - atot);
        low = min(low, top);
        if (K.schedule != 0) {
            // asynchronous schedule: a finished rollout returns its slot, and the prompt whose
            // batch it completes is listed for the decisions at this step boundary
            const int fin = (i < live && !keep) ? 1 : 0;
            int stot;
            const int soff = scan256(fin, stot, warp_tot);
            if (fin) {
                c.slot_free[stop + soff] = slot;
                const int q = c.seq_q[slot];
                if (atomicSub(&c.q_inflight[q], 1) == 1) c.dec_list[atomicAdd(&V.n_dec, 1)] = q;
            }
            stop += stot;
        }
        // stable in-place compaction: a kept row lands at or before its own index
        int tot;
        const int before = scan256(keep, tot, warp_tot);
        if (keep) {
            const int dst = out + before;
            c.row_slot[dst] = slot;
            c.row_pos[dst] = Lp - 1 + gen;
            c.row_tok[dst] = next_tok;
            c.row_seed[dst] = sampler_row_seed(K.sample_seed, c.seq_uid[slot], gen);
        }
        __syncthreads();
        out += tot;
    }
    // attention items of the next step: splits of `span` KV blocks
    const int span = att_span_rows(c.row_pos, out, K, span_sm);
    int items = 0;
    for (int base = 0; base < out; base += 256) {
        const int i = base + tid;
        const int ns = (i < out) ? ((c.row_pos[i] + K.attn_chunk) / K.attn_chunk + span - 1) / span : 0;
        int tot;
        const int before = scan256(ns, tot, warp_tot);
        if (i < out) {
            const int i0 = items + before;
            c.row_item0[i] = i0;
            for (int sp = 0; sp < ns; ++sp) {
                if (i0 + sp < c.att_cap) c.att_items[i0 + sp] = make_int2(i, sp);
                else report_error(&V.err, ERR_CAPACITY);
            }
        }
        items += tot;
    }
    if (tid == 0) {
        V.live = out;
        V.att_items = min(items, c.att_cap);
        V.att_span = span;
        V.exec_steps += 1;
        V.round_steps += 1;
        V.blk_top = top;
        V.blk_low = low;
        V.slot_top = stop;
        if (use_more) {
            bool next = out > 0 && *(volatile int *)&V.err == 0 &&
                        (K.schedule != 0 ? V.n_dec == 0 && V.exec_steps <= (int64_t)K.N * K.max_gen + 1
                                         : V.round_steps <= V.round_maxL);
            if (next) {  // one more iteration of the loop
                V.iters += 1;
                if (K.max_iters > 0 && V.iters > K.max_iters) {
                    report_error(&V.err, ERR_ITER_BOUND);
                    next = false;
                }
            }
            cudaGraphSetConditional(more, next ? 1u : 0u);
        }
    }
}

// Teacher forcing: n rollouts, rollout i uses prompt slot i and rollout slot i, lengths T.
static __global__ void __launch_bounds__(kCtlThreads, 1) teacher_setup_kernel(StepPtrs c, int n, const int64_t *uid) {
    pdl_wait_prior_grids();
    const StepConst &K = *c.kc;
    StepVars &V = *c.v;
    const int Lp = K.Lp, Lpre = Lp - 1;
    const int nblk = (Lp + K.attn_chunk - 1) / K.attn_chunk;
    const int span = att_span_uniform(n, nblk, K.att_kvh, K.att_ctas);
    const int nsplit = (nblk + span - 1) / span;
    const int nsh = shared_blocks(Lp, K.attn_chunk);
    for (int i = threadIdx.x; i < c.n_priv; i += kCtlThreads) c.blk_free[i] = c.n_shared + c.n_priv - 1 - i;
    __syncthreads();
    for (int r = threadIdx.x; r < n; r += kCtlThreads) {
        int32_t *bt = c.blk_tab + (int64_t)r * c.nblk_max;  // prompt r's full blocks, then a private one
        for (int j = 0; j < nsh; ++j) bt[j] = r * c.nsh_max + j;
        bt[nsh] = r < c.n_priv ? c.blk_free[c.n_priv - 1 - r] : c.n_shared;  // (n > n_priv: an error)
        c.fresh_pslot[r] = r;
        c.new_slots[r] = r;
        c.seq_q[r] = r;
        c.seq_j[r] = 0;
        c.seq_len[r] = K.T_forced;
        c.seq_gen[r] = 0;
        c.seq_pslot[r] = r;
        c.seq_uid[r] = uid[r];
        c.row_slot[r] = r;
        c.row_pos[r] = Lp - 1;
        c.row_tok[r] = c.p_tok[(int64_t)r * Lp + Lp - 1];
        c.row_seed[r] = sampler_row_seed(K.sample_seed, uid[r], 0);
        c.row_item0[r] = r * nsplit;
        for (int sp = 0; sp < nsplit; ++sp) c.att_items[r * nsplit + sp] = make_int2(r, sp);
    }
    for (int r = threadIdx.x; r < n * Lpre; r += kCtlThreads) {
        const int f = r / Lpre, t = r - f * Lpre;
        c.pre_slot[r] = f;
        c.pre_pos[r] = t;
        c.pre_tok[r] = c.p_tok[(int64_t)f * Lp + t];
    }
    if (threadIdx.x == 0) {
        StepVars z;
        memset(&z, 0, sizeof(z));
        z.round = 0;
        z.live = n;
        z.att_items = n * nsplit;
        z.att_span = span;
        z.pre_rows = n * Lpre;
        z.n_fresh = n;
        z.round_maxL = K.T_forced;
        z.kt0 = ~0ull;
        z.blk_top = z.blk_low = c.n_priv - n;
        z.n_new = n;
        if (n > c.n_priv) z.err |= ERR_CAPACITY;
        V = z;
    }
}

// Gumbel-max over given fp32 logits (kernel-level entry point), short vocabularies: one CTA per row, the
// noise of every token.  Bound by the CTAs' latency chain, where the bounds of sample_rows_kernel cost more than
// the logarithms they save: 65,536 rows x 512: 148 us against 426, 4,096 x 2,048 29 against 36,
// 4,096 x 4,096 49 against 47.
constexpr int kSampleShort = 2048;
static __global__ void __launch_bounds__(256) sample_short_rows_kernel(const float *logits, int V, uint64_t sample_seed,
                                                                       const int64_t *uid, const int32_t *t, int *token) {
    __shared__ float sv[8];
    __shared__ int si[8];
    const int r = blockIdx.x;
    const uint64_t rs = sampler_row_seed(sample_seed, uid[r], t[r]);
    float best = -INFINITY;
    int bi = 0x7fffffff;
    for (int v = threadIdx.x; v < V; v += 256) {
        const float z = __fadd_rn(logits[(int64_t)r * V + v], gumbel_from_hash(splitmix_at(rs, (uint64_t)v + 1)));
        if (z > best) { best = z; bi = v; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
    }
    if ((threadIdx.x & 31) == 0) { sv[threadIdx.x >> 5] = best; si[threadIdx.x >> 5] = bi; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w)
            if (sv[w] > best || (sv[w] == best && si[w] < bi)) { best = sv[w]; bi = si[w]; }
        token[r] = bi;
    }
}

// Longer vocabularies: 1 to 8 CTAs per row (sample_ctas, a cluster), each a contiguous share of the
// vocabulary, the row's maximum joined through distributed shared memory.  Bound by instruction issue (a
// 64-bit hash per token; 54 instructions a token in all), so the noise's logarithms are taken only for tokens
// that could reach the CTA's best so far (noise_cut), the hash's input is advanced by additions, and a step's
// logits load during the one before.  64 rows x 151,936, whole call: 27 us (kernel 25), 277 us with one CTA per
// row (64 of 152 SMs) and the noise of every token.
constexpr int kSampleCtas = 8;
// The split doubles while a CTA would still hold more than a thousand tokens and the CTAs fit the SMs at
// once (8 an SM): a cluster costs ~48 ns of launch, so rows that fill the SMs by themselves take one CTA each
// and no cluster (4,096 rows x 4,096: 212 us in clusters of 8, 47 without).
inline int sample_ctas(int R, int V, int sms) {
    int n = 1;
    while (n < kSampleCtas && V > 1024 * n && (int64_t)R * 2 * n <= (int64_t)8 * sms) n *= 2;
    return n;
}
static __global__ void __launch_bounds__(256) sample_rows_kernel(const float *logits, int V, uint64_t sample_seed,
                                                                 const int64_t *uid, const int32_t *t, int *token,
                                                                 int ctas) {
    __shared__ float sv[8];
    __shared__ int si[8];
    __shared__ uint32_t cv[kSampleCtas], ci[kSampleCtas];  // (rank 0) the cluster's maxima
    __shared__ volatile float wb[8];                       // each warp's best so far
    if (ctas > 1) cluster_arrive();  // (waited for before the store into rank 0's shared memory)
    if (threadIdx.x < 8) wb[threadIdx.x] = -INFINITY;
    __syncthreads();
    const int r = blockIdx.x / ctas, rank = (int)(blockIdx.x - (unsigned)r * ctas);
    const uint64_t rs = sampler_row_seed(sample_seed, uid[r], t[r]);
    // this CTA's share: n tokens from tok0 on (n < 2^29: rows of more fit no memory in such numbers that
    // they get one CTA each)
    const int64_t per = (((int64_t)V - 1) / ctas + 4) & ~(int64_t)3, tok0 = rank * per;
    const int n = (int)max((int64_t)0, min(V - tok0, per));
    const float *row = logits + (int64_t)r * V + tok0;
    const bool vec = (reinterpret_cast<uintptr_t>(row) & 15) == 0;
    float best = -INFINITY, wbest = -INFINITY;  // this thread's, and the warp's as of the last step
    int bi = 0x7fffffff;
    bool first = true;
    // a step's tokens: b + 4 tid .. and b + 1024 + 4 tid ..
    auto load = [&](int b, float (&y)[8]) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int v = b + q * 1024 + (int)threadIdx.x * 4;
            if (vec && v + 3 < n) {
                const float4 x = __ldg(reinterpret_cast<const float4 *>(row + v));
                y[4 * q] = x.x; y[4 * q + 1] = x.y; y[4 * q + 2] = x.z; y[4 * q + 3] = x.w;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) y[4 * q + e] = v + e < n ? __ldg(row + v + e) : -INFINITY;
            }
        }
    };
    float next[8];
    load(0, next);
#pragma unroll 1
    for (int b = 0; b < n; b += 2048) {
        float z[8];
        uint32_t cand = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) z[e] = next[e];
        if (n - b > 2048) load(b + 2048, next);  // (in flight during this step)
        // the hash's input is linear in the token: one product per four of them
        uint32_t code[8];  // the hash's top 24 bits
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint64_t v = (uint64_t)tok0 + (uint32_t)(b + q * 1024) + threadIdx.x * 4;
            const uint64_t x = rs + (v + 1) * kSplitmixGamma;
#pragma unroll
            for (int e = 0; e < 4; ++e) code[4 * q + e] = (uint32_t)(mix64(x + (uint64_t)e * kSplitmixGamma) >> 40);
        }
        const int n0 = n - b - (int)threadIdx.x * 4, n1 = n0 - 1024;  // this thread's tokens of each four
        const uint32_t valid = (n0 >= 4 ? 0xfu : n0 > 0 ? (1u << n0) - 1 : 0u) | (n1 >= 4 ? 0xf0u : n1 > 0 ? (16u << n1) - 16 : 0u);
        if (first) {  // before the first maximum, the warp's best of the tokens of largest noise stands in for it
            first = false;
            uint32_t most = 0;
            float zmost = -INFINITY;
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (code[e] >= most && (valid >> e & 1)) { most = code[e]; zmost = z[e]; }
            wbest = __fadd_rn(zmost, gumbel_from_hash((uint64_t)most << 40));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) wbest = fmaxf(wbest, __shfl_xor_sync(0xffffffffu, wbest, o));
        }
        float vmax = z[0];
#pragma unroll
        for (int e = 1; e < 8; ++e) vmax = fmaxf(vmax, z[e]);
        const uint32_t thr = noise_cut(wbest, vmax);
#pragma unroll
        for (int e = 0; e < 8; ++e) cand |= (uint32_t)(code[e] >= thr) << e;
        cand &= valid;
#pragma unroll 1
        while (cand) {  // in increasing token order: the first maximum is kept
            const int e = __ffs(cand) - 1;
            cand &= cand - 1;
            float ze = z[0];
            uint32_t k = code[0];
#pragma unroll
            for (int i = 1; i < 8; ++i) {
                ze = (i == e) ? z[i] : ze;
                k = (i == e) ? code[i] : k;
            }
            const int v = (int)tok0 + b + (e >> 2) * 1024 + (int)threadIdx.x * 4 + (e & 3);
            ze = __fadd_rn(ze, gumbel_from_hash((uint64_t)k << 40));  // (the noise is of the top 24 bits)
            if (ze > best) { best = ze; bi = v; }
        }
        // the next step's bound: the CTA's best so far (a warp that is behind reads an older one)
        wbest = fmaxf(wbest, best);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wbest = fmaxf(wbest, __shfl_xor_sync(0xffffffffu, wbest, o));
        if ((threadIdx.x & 31) == 0) wb[threadIdx.x >> 5] = wbest;
        __syncwarp();
        for (int w = 0; w < 8; ++w) wbest = fmaxf(wbest, wb[w]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    if ((threadIdx.x & 31) == 0) { sv[threadIdx.x >> 5] = best; si[threadIdx.x >> 5] = bi; }
    __syncthreads();
    if (ctas > 1) cluster_wait();  // every CTA of the cluster has started
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w)
            if (sv[w] > best || (sv[w] == best && si[w] < bi)) { best = sv[w]; bi = si[w]; }
        if (ctas == 1) {
            token[r] = bi;
        } else {
            st_cluster_u32(cluster_addr(&cv[rank], 0), __float_as_uint(best));
            st_cluster_u32(cluster_addr(&ci[rank], 0), (uint32_t)bi);
        }
    }
    if (ctas == 1) return;
    cluster_sync();
    if (rank == 0 && threadIdx.x == 0) {
        best = -INFINITY;
        bi = 0x7fffffff;
        for (int w = 0; w < ctas; ++w) {
            const float ov = __uint_as_float(cv[w]);
            if (ov > best || (ov == best && (int)ci[w] < bi)) { best = ov; bi = (int)ci[w]; }
        }
        token[r] = bi;
    }
}

}  // namespace sara
