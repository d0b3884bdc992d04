"""Edges of the kernel-level row operations: the sampler's cluster shares and unaligned rows, the projection GEMM's K
splits and tile walks, the attention's position shares, alignment and refusals."""
import numpy as np
import pytest

import synth
from gpu_util import assert_drawn_by_the_rule
from oracle import decode as o2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_26253_gb300 as p
    p.load()
    return p


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# vocabularies around the shares of a row's 8 CTAs (multiples of 4 tokens, 2,048 a step); odd ones leave rows unaligned
@pytest.mark.parametrize("V", [1, 5, 31, 32, 33, 512, 2047, 8191, 32001, 131073])
def test_sampler_vocabulary_edges(pkg, V):
    rng = np.random.default_rng(V)
    R = 5
    logits = (rng.standard_normal((R, V)) * 2).astype(np.float32)
    uid, t = np.arange(R, dtype=np.int64) * 7 + 1, np.arange(R, dtype=np.int32) * 3
    tok = pkg.sample(_dev(logits), _dev(uid), _dev(t), 11).cpu().numpy()
    for r in range(R):
        want, margin = o2.sample_token(logits[r], 11, int(uid[r]), int(t[r])) if V > 1 else (0, 1.0)
        if margin > 1e-5:
            assert tok[r] == want, (r, tok[r], want, margin)


# the largest vocabulary whose token ids are 32-bit: shares and their steps end within 2,048 of 2^31
@pytest.mark.parametrize("V", [2 ** 31 - 1, 2 ** 31 - 900])
def test_sampler_largest_vocabulary(pkg, V):
    import torch
    per = (-(-V // 8) + 3) // 4 * 4
    logits = torch.full((1, V), -np.inf, device="cuda")
    one = torch.ones(1, dtype=torch.int64, device="cuda")
    for v in (0, per - 1, 7 * per, V - 1):
        logits[0, v] = 0
        assert int(pkg.sample(logits, one, one.int(), 4)) == v
        logits[0, v] = -np.inf


# many rows of few tokens; the lines between the kernels and of the split: 8, 4, 2 and 1 CTAs a row, the last with few
# tokens, so that it reaches the join of the maxima at once
@pytest.mark.parametrize("R,V", [(6000, 1), (6000, 40), (1, 2048), (1, 2049), (1, 4097), (152, 8193), (153, 8193),
                                 (304, 2049), (305, 2049), (609, 2050)])
def test_sampler_rows_and_splits(pkg, R, V):
    rng = np.random.default_rng(V)
    logits = (rng.standard_normal((R, V)) * 2).astype(np.float32)
    uid, t = np.arange(R, dtype=np.int64), np.zeros(R, np.int32)
    tok = pkg.sample(_dev(logits), _dev(uid), _dev(t), 4).cpu().numpy()
    assert tok.min() >= 0 and tok.max() < V
    for r in range(R if V > 1 else 0):
        want, margin = o2.sample_token(logits[r], 4, r, 0)
        if margin > 1e-5:
            assert tok[r] == want, (r, tok[r], want, margin)


def test_sampler_most_rows(pkg):
    # more rows than a grid holds clusters of 8 CTAs
    import torch
    R = 2 ** 28 + 5
    uid, t = torch.arange(R, device="cuda"), torch.zeros(R, dtype=torch.int32, device="cuda")
    tok = pkg.sample(torch.zeros((R, 1), device="cuda"), uid, t, 4)
    assert int(tok.min()) == 0 and int(tok.max()) == 0


# logits so large that the sum with the noise is rounded (spacing 0.008 to 0.06), equal or nearly so: the token that
# bounds the others keeps its place, and ties go to the lowest id
@pytest.mark.parametrize("V", [512, 5000, 40003])
@pytest.mark.parametrize("mean,std", [(65536.0, 0.0), (65536.0, 1.0), (-65536.0, 1.0), (1e6, 0.0), (1e6, 1.0)])
def test_sampler_large_logits(pkg, V, mean, std):
    rng = np.random.default_rng(V)
    R = 60
    logits = (mean + std * rng.standard_normal((R, V))).astype(np.float32)
    tok = pkg.sample(_dev(logits), _dev(np.arange(R, dtype=np.int64)), _dev(np.zeros(R, np.int32)), 5).cpu().numpy()
    clear = sum(assert_drawn_by_the_rule(tok[r], logits[r], 5, r, 0) for r in range(R))
    assert clear >= R * 3 // 4


def test_sampler_infinities_and_nan(pkg):
    V, R = 4099, 4
    logits = np.full((R, V), -np.inf, np.float32)
    logits[1, [17, 4000]] = np.inf           # the first infinity wins
    logits[2, 3001] = -1e30                  # the only finite logit
    logits[3, ::2] = np.nan                  # a NaN is never drawn
    logits[3, 1::2] = 0.0
    uid, t = np.arange(R, dtype=np.int64), np.zeros(R, np.int32)
    tok = pkg.sample(_dev(logits), _dev(uid), _dev(t), 3).cpu().numpy()
    assert tok[0] == 0x7FFFFFFF and tok[1] == 17 and tok[2] == 3001 and tok[3] % 2 == 1


# one tile: K splits 1, 2, 4 and 8, uneven shares; tile counts at which the split halves, up to 64 rows and above (other
# CTAs per SM); more tiles than CTAs
@pytest.mark.parametrize("R,N,K", [(1, 128, 64), (31, 128, 128), (32, 128, 448), (33, 128, 1088), (128, 4864, 640),
                                   (5, 4992, 640), (64, 9856, 320), (65, 19584, 192), (127, 40064, 192),
                                   (65, 128, 704), (97, 1920, 1088), (96, 4352, 640), (72, 9728, 640), (70, 9856, 640)])
@pytest.mark.parametrize("static", [False, True])
def test_gemm_splits_and_tile_walks(pkg, R, N, K, static):
    import torch
    rng = np.random.default_rng(R + N + K)
    X = synth.f32_to_bf16_bits(rng.standard_normal((R, K)).astype(np.float32))
    W = synth.f32_to_bf16_bits((rng.standard_normal((N, K)) * 0.02).astype(np.float32))
    f = pkg.gemm_bf16_static if static else pkg.gemm_bf16
    Y = f(_dev(X.view(np.int16)).view(torch.bfloat16), _dev(W.view(np.int16)).view(torch.bfloat16)).cpu().numpy()
    xf, wf = synth.bf16_bits_to_f32(X).astype(np.float64), synth.bf16_bits_to_f32(W).astype(np.float64)
    # fp32 accumulation of exact bf16 products: |error| <= K 2^-23 sum |x w|
    bound = K * 2.0 ** -23 * (np.abs(xf) @ np.abs(wf).T) + 1e-6
    assert (np.abs(Y - xf @ wf.T) <= bound).all()


# The tensor core's accumulation truncates: about 1e-9 of the result per element of K in one chain (1.25e-9 allowed), so
# chains are cut to half of what an even split over the SMs gives one, 64 elements at least; beyond that only the result
# is rounded (2^-24).
@pytest.mark.parametrize("R,N,K", [(8, 128, 2368), (100, 256, 4096), (4, 2048, 1536), (128, 2048, 1536), (16, 2048, 11008),
                                   (15, 1536, 8960), (33, 17920, 1536), (64, 40064, 1536), (128, 40064, 1536), (3, 19584, 9024)])
def test_gemm_accumulation_chains(pkg, R, N, K):
    import torch
    g = torch.Generator(device="cuda").manual_seed(N + K)
    X = torch.randn((R, K), generator=g, device="cuda").bfloat16()
    W = torch.randn((N, K), generator=g, device="cuda").bfloat16()
    want = X.double() @ W.double().t()
    chain = max(1, min(K // 64, N // 128 * (K // 64) // torch.cuda.get_device_properties(0).multi_processor_count) // 2)
    rel = float((pkg.gemm_bf16(X, W).double() - want).norm() / want.norm())
    assert rel < 1.25e-9 * 64 * chain + 2.0 ** -24, (rel, chain)


# infinite and NaN activations and sums past the largest float: the same results with K split over a cluster and not
@pytest.mark.parametrize("N,K", [(128, 128), (256, 1088), (2048, 1536), (40064, 192)])
def test_gemm_infinities_and_nan(pkg, N, K):
    import torch
    rng = np.random.default_rng(N + K)
    X = torch.from_numpy(rng.standard_normal((6, K)).astype(np.float32)).bfloat16().cuda()
    W = torch.from_numpy(rng.uniform(0.5, 1.0, (N, K)).astype(np.float32)).bfloat16().cuda()
    W[1::2] *= -1
    X[1, 5], X[2, K - 1], X[3, 7], X[3, K - 7], X[4, K // 2] = np.inf, -np.inf, np.inf, np.inf, np.nan
    X[5] = 3e38  # every partial sum overflows
    Y = pkg.gemm_bf16(X, W).cpu()
    sign = torch.ones(N)
    sign[1::2] = -1
    want = X[:1].double().cpu() @ W.double().cpu().t()
    assert torch.allclose(Y[:1].double(), want, rtol=1e-4, atol=1e-3)
    for r, s in ((1, 1), (2, -1), (3, 1), (5, 1)):
        assert torch.equal(Y[r], s * sign * np.inf), r
    assert Y[4].isnan().all()


def _attention_ref(q, kv, ctx, n_kv):
    b, H, hd = q.shape
    out = np.zeros((b, H, hd))
    for i in range(b):
        for h in range(H):
            K, V = kv[i, 0, h // (H // n_kv), :ctx[i]], kv[i, 1, h // (H // n_kv), :ctx[i]]
            s = K @ q[i, h] / np.sqrt(hd)
            p = np.exp(s - s.max())
            out[i, h] = (p / p.sum()) @ V
    return out


def _attention_case(rng, H, KVH, hd, ctxs):
    b, cap = len(ctxs), max(ctxs) + 3
    return (rng.standard_normal((b, H, hd)).astype(np.float16), rng.standard_normal((b, 2, KVH, cap, hd)).astype(np.float16),
            np.array(ctxs, np.int32), cap)


def _check_attention(out, q, kv, ctx, KVH):
    import torch
    got = synth.bf16_bits_to_f32(out.view(torch.int16).cpu().numpy().view(np.uint16)).astype(np.float64)
    want = _attention_ref(q.astype(np.float64), kv.astype(np.float64), ctx, KVH)
    # the bf16 rounding of the output (2^-9 relative) dominates
    assert np.all(np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 1e-3)


# positions around a warp's step of 16 and the CTAs' shares of a row; every group size and head dim; one row and many
@pytest.mark.parametrize("H,KVH,hd,ctxs", [(6, 1, 128, [1]), (8, 1, 64, [15, 16, 17]), (2, 1, 32, [63, 64, 65, 129]),
                                          (4, 4, 128, [512, 1, 513]), (8, 2, 32, [2048, 7]),
                                          (12, 2, 128, list(range(1, 101))), (16, 2, 64, [12288])])
def test_attention_edges(pkg, H, KVH, hd, ctxs):
    q, kv, ctx, cap = _attention_case(np.random.default_rng(H + hd), H, KVH, hd, ctxs)
    out = pkg.attention_decode(_dev(q), _dev(kv), _dev(ctx), KVH, cap, max_ctx=max(ctxs))
    _check_attention(out, q, kv, ctx, KVH)


def test_attention_unaligned_operands(pkg):
    # q and K / V that start 8 bytes off a 16-byte boundary (head dim 64): accepted as ever
    import torch
    q, kv, ctx, cap = _attention_case(np.random.default_rng(1), 8, 2, 64, [100, 300])

    def off(a):
        buf = torch.zeros(a.size + 4, dtype=torch.float16, device="cuda")
        buf[4:] = _dev(a).reshape(-1)
        return buf[4:].view(a.shape)

    _check_attention(pkg.attention_decode(off(q), off(kv), _dev(ctx), 2, cap), q, kv, ctx, 2)


@pytest.mark.parametrize("hd,elements", [(128, 4), (64, 2), (32, 1)])
def test_attention_operands_below_their_loads_alignment_refused(pkg, hd, elements):
    # a head dim's rows are read hd / 16 elements at a time: less alignment is an error, not a fault
    import torch
    q = torch.zeros(2 * 4 * hd + 8, dtype=torch.float16, device="cuda")[elements:][:2 * 4 * hd].view(2, 4, hd)
    kv = torch.zeros((2, 2, 2, 20, hd), dtype=torch.float16, device="cuda")
    ctx = torch.full((2,), 20, dtype=torch.int32, device="cuda")
    with pytest.raises(pkg.SaraError) as e:
        pkg.attention_decode(q, kv, ctx, 2, 20)
    assert e.value.code == pkg.SARA_EINVAL


def test_attention_infinite_value(pkg):
    # an infinite V element reaches the result with its sign, beside exact values in the other dims
    q, kv, ctx, cap = _attention_case(np.random.default_rng(2), 12, 2, 128, [40, 300])
    kv[0, 1, 0, 7, 5], kv[1, 1, 1, 250, 90] = np.inf, -np.inf
    out = pkg.attention_decode(_dev(q), _dev(kv), _dev(ctx), 2, cap).float().cpu().numpy()
    assert np.all(out[0, :6, 5] == np.inf) and np.all(out[1, 6:, 90] == -np.inf)
    mask = np.isfinite(out)
    assert mask.sum() == out.size - 12
    kv[~np.isfinite(kv)] = 0
    want = _attention_ref(q.astype(np.float64), kv.astype(np.float64), ctx, 2)
    assert np.all(np.abs(out - want)[mask] <= 2.0 ** -8 * np.abs(want)[mask] + 2e-3)


def test_attention_infinite_value_of_small_probability(pkg):
    # position 0 outweighs the others by e^40: their probabilities (2^-58) are far below what fp16 holds
    q = np.ones((1, 8, 128), np.float16)
    kv = np.zeros((1, 2, 1, 303, 128), np.float16)
    kv[0, 0, 0, 0], kv[0, 1] = 40 / np.sqrt(128), np.random.default_rng(5).standard_normal((1, 303, 128))
    want = kv[0, 1, 0, 0].astype(np.float32)
    kv[0, 1, 0, 3, 17], kv[0, 1, 0, 299, 90] = np.inf, -np.inf  # in the same warp's step, in another CTA
    out = pkg.attention_decode(_dev(q), _dev(kv), _dev(np.array([300], np.int32)), 1, 303).float().cpu().numpy()[0]
    assert np.all(out[:, 17] == np.inf) and np.all(out[:, 90] == -np.inf)
    mask = np.isfinite(out[0])
    assert mask.sum() == 126 and np.all(np.abs(out - want)[:, mask] <= 2.0 ** -8 * np.abs(want)[mask])


def test_attention_infinite_value_beside_cancelling_ones(pkg):
    # values of +-1000 under nearly equal probabilities cancel to ~0.06: the other dims of a row with an infinite value
    # need all of the probabilities' 24 bits (1000 * 2^-24 of each of 300, averaged: below 1e-5)
    q, kv, ctx, cap = _attention_case(np.random.default_rng(6), 6, 1, 128, [300])
    q *= np.float16(0.001)
    kv[0, 1] = np.where(np.arange(cap) % 2 == 0, 1000, -1000).astype(np.float16)[None, :, None]
    want = _attention_ref(q.astype(np.float64), kv.astype(np.float64), ctx, 1)
    kv[0, 1, 0, 7, 5] = np.inf
    out = pkg.attention_decode(_dev(q), _dev(kv), _dev(ctx), 1, cap).float().cpu().numpy()
    assert np.all(out[0, :, 5] == np.inf)
    mask = np.arange(128) != 5
    assert np.all(np.abs(out - want)[..., mask] <= 2.0 ** -8 * np.abs(want)[..., mask] + 1e-4)


@pytest.mark.parametrize("bad", [0, -1, 301])
def test_attention_context_out_of_range_refused(pkg, bad):
    q, kv, ctx, cap = _attention_case(np.random.default_rng(3), 4, 2, 32, [300, 20, 5])
    ctx[1] = bad
    with pytest.raises(pkg.SaraError) as e:
        pkg.attention_decode(_dev(q), _dev(kv), _dev(ctx), 2, cap, max_ctx=300)
    assert e.value.code == pkg.SARA_EINVAL


@pytest.mark.parametrize("where", [0, 1700, 2999])
def test_attention_refused_call_writes_nothing(pkg, where):
    import torch
    b, H, KVH, hd, cap = 3000, 4, 2, 32, 70
    q = torch.ones((b, H, hd), dtype=torch.float16, device="cuda")
    kv = torch.ones((b, 2, KVH, cap, hd), dtype=torch.float16, device="cuda")
    ctx = torch.full((b,), 64, dtype=torch.int32, device="cuda")
    ctx[where] = 71
    out = torch.full((b, H, hd), 7.0, dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(pkg.load().sara_attention_workspace_bytes(b, H, hd, cap), dtype=torch.uint8, device="cuda")

    def call():
        return pkg.load().sara_attention_decode(q.data_ptr(), kv.data_ptr(), kv.stride(0), ctx.data_ptr(), out.data_ptr(), b,
                                                H, KVH, hd, cap, cap, ws.data_ptr(), ws.numel(),
                                                torch.cuda.current_stream().cuda_stream)
    assert call() == pkg.SARA_EINVAL and bool((out == 7).all())
    ctx[where] = 64
    assert call() == pkg.SARA_OK and bool((out == 1).all())
