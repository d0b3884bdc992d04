"""Edges of the kernel-level row operations: the sampler's cluster shares and unaligned rows, the projection GEMM's K
splits and tile walks."""
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


# one tile: K splits 1, 2, 4 and 8, uneven shares; tile counts at which the split halves; more tiles than CTAs
@pytest.mark.parametrize("R,N,K", [(1, 128, 64), (31, 128, 128), (32, 128, 448), (33, 128, 1088), (128, 4864, 640),
                                   (5, 4992, 640), (64, 9856, 320), (65, 19584, 192), (127, 40064, 192)])
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
