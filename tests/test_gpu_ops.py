"""Kernel-level parity through the C ABI: the tcgen05 projection GEMM, decode attention and
the Gumbel-max sampler against the float64 / float32 oracle on the same inputs."""
import numpy as np
import pytest

import synth
from oracle import decode as o2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_26253_gb300 as p
    p.load()
    return p


def _bf16(rng, shape, scale=1.0):
    return synth.f32_to_bf16_bits((rng.standard_normal(shape) * scale).astype(np.float32))


def _dev(a):
    import torch
    t = torch.from_numpy(np.ascontiguousarray(a.view(np.int16) if a.dtype == np.uint16 else a))
    return t.cuda()


def _dev_bf16(a):
    import torch
    return _dev(a).view(torch.bfloat16)


@pytest.mark.parametrize("R,N,K", [(1, 128, 64), (7, 384, 128), (25, 1536, 1536), (64, 2048, 1536),
                                   (128, 1536, 8960), (33, 17920, 1536), (128, 256, 4096), (16, 151936, 1536),
                                   (100, 128, 11008)])
def test_gemm_matches_float64(pkg, R, N, K):
    rng = np.random.default_rng(R * 1000 + N + K)
    X = _bf16(rng, (R, K))
    W = _bf16(rng, (N, K), 0.02)
    Y = pkg.gemm_bf16(_dev_bf16(X), _dev_bf16(W)).cpu().numpy()
    xf = synth.bf16_bits_to_f32(X).astype(np.float64)
    wf = synth.bf16_bits_to_f32(W).astype(np.float64)
    want = xf @ wf.T
    # fp32 accumulation of exact bf16 products: |error| <= K 2^-23 sum |x w|
    bound = K * 2.0 ** -23 * (np.abs(xf) @ np.abs(wf).T) + 1e-6
    bad = np.abs(Y - want) > bound
    assert not bad.any(), (np.argwhere(bad)[:5], Y[bad][:5], want[bad][:5])


def test_gemm_repeated_calls_reuse_workspace(pkg):
    import torch
    rng = np.random.default_rng(5)
    X = _dev_bf16(_bf16(rng, (40, 1536)))
    W = _dev_bf16(_bf16(rng, (1536, 1536), 0.02))
    ws = torch.zeros(pkg.load().sara_gemm_workspace_bytes(40, 1536, 1536), dtype=torch.uint8, device="cuda")
    a = pkg.gemm_bf16(X, W, workspace=ws)
    b = pkg.gemm_bf16(X, W, workspace=ws)
    assert torch.equal(a, b)  # the same sums on every run


def _attention_ref(q, kv, ctx, n_kv):
    """float64 softmax(q K^T / sqrt(hd)) V over positions < ctx per row (GQA)."""
    b, H, hd = q.shape
    G = H // n_kv
    out = np.zeros((b, H, hd))
    for i in range(b):
        for h in range(H):
            K = kv[i, 0, h // G, :ctx[i]]
            V = kv[i, 1, h // G, :ctx[i]]
            s = K @ q[i, h] / np.sqrt(hd)
            p = np.exp(s - s.max())
            out[i, h] = (p / p.sum()) @ V
    return out


@pytest.mark.parametrize("hd,H,KVH,ctxs", [(128, 12, 2, [1, 17, 256, 257, 1000]),
                                          (128, 16, 2, [4096, 300, 2]),
                                          (32, 4, 2, [1, 31, 64, 513]),
                                          (64, 8, 8, [100, 255]),
                                          (128, 8, 2, [8576, 129])])
def test_attention_matches_float64(pkg, hd, H, KVH, ctxs):
    import torch
    rng = np.random.default_rng(hd + H + len(ctxs))
    b = len(ctxs)
    cap = max(ctxs) + 16
    q = rng.standard_normal((b, H, hd)).astype(np.float16)
    kv = rng.standard_normal((b, 2, KVH, cap, hd)).astype(np.float16)
    ctx = np.array(ctxs, np.int32)
    out = pkg.attention_decode(torch.from_numpy(q).cuda(), torch.from_numpy(kv).cuda(), _dev(ctx), KVH, cap)
    got = synth.bf16_bits_to_f32(out.view(torch.int16).cpu().numpy().view(np.uint16)).astype(np.float64)
    want = _attention_ref(q.astype(np.float64), kv.astype(np.float64), ctx, KVH)
    # the bf16 rounding of the output (2^-9 relative) dominates
    assert np.all(np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 1e-3)


def test_sampler_matches_oracle_gumbel_max(pkg):
    rng = np.random.default_rng(9)
    R, V = 24, 151936
    logits = (rng.standard_normal((R, V)) * 2).astype(np.float32)
    uid = np.arange(R, dtype=np.int64) * 64 + 3
    t = (np.arange(R, dtype=np.int32) * 37) % 4096
    tok = pkg.sample(_dev(logits), _dev(uid), _dev(t), 5).cpu().numpy()
    checked = 0
    for r in range(R):
        want, margin = o2.sample_token(logits[r], 5, int(uid[r]), int(t[r]))
        if margin > 1e-5:
            assert tok[r] == want, (r, tok[r], want, margin)
            checked += 1
    assert checked >= R - 2
