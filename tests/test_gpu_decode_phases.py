"""The decode step's row-count and width branches: every accumulator layout of its projections (row counts around 8, 16,
32, 64 and 128), MLP widths and vocabularies from a single 16-feature unit per CTA to more than one 256-feature pass, more
attention units than a CTA's table holds, new positions at the edges of a warp's 32 positions and of a KV block (where the
number of attention splits changes); teacher-forced logits against the float64 oracle within the stated tolerance."""
import numpy as np
import pytest

import synth
from gpu_util import LOGIT_MAX_ABS, LOGIT_REL_L2, assert_drawn_by_the_rule, logit_errors
from oracle import decode as o2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2607_26253_gb300 as p
    p.load()
    return p


def _shape(name, **kw):
    base = dict(layers=2, d_model=256, n_heads=4, n_kv_heads=2, head_dim=64, ffn=320, vocab=640)
    base.update(kw)
    return synth.ModelShape(name, **base)


NARROW = _shape("ffn 64", d_model=128, n_heads=4, head_dim=32, ffn=64)
ODD = _shape("ffn 320")
WIDE = _shape("ffn 20032", layers=1, ffn=20032)                     # 2,504 units: two passes on some CTAs
DEEP = _shape("d 2048", layers=2, d_model=2048, n_heads=16, head_dim=128, ffn=448)
ODD_D = _shape("d 1664", layers=1, d_model=1664, n_heads=4, head_dim=128, ffn=128)  # 26 units of 64: 1,222 at 47 rows
MANY_HEADS = _shape("32 heads", d_model=512, n_heads=32, n_kv_heads=4, head_dim=128, ffn=128)  # K = 4,096 > d
MANY_KV = _shape("48 kv heads", layers=2, d_model=128, n_heads=48, n_kv_heads=48, head_dim=32, ffn=64)  # 40 units per SM
VOCAB_UNITS = _shape("vocab 40064", layers=1, d_model=128, n_heads=4, head_dim=32, ffn=64, vocab=40064)  # 2,504 units
VOCAB_TILES = _shape("vocab 80000", layers=1, d_model=128, n_heads=4, head_dim=32, ffn=64, vocab=80000)  # whole tiles


@pytest.mark.parametrize("shape,rows", [(NARROW, 1), (NARROW, 9), (NARROW, 128), (ODD, 8), (ODD, 17), (ODD, 33),
                                        (ODD, 65), (WIDE, 2), (WIDE, 32), (WIDE, 64), (DEEP, 1), (DEEP, 16),
                                        (DEEP, 31), (DEEP, 48), (ODD_D, 47), (MANY_HEADS, 3), (MANY_HEADS, 32), (MANY_HEADS, 40),
                                        (MANY_KV, 128), (VOCAB_UNITS, 3), (VOCAB_UNITS, 66),
                                        (VOCAB_TILES, 3), (VOCAB_TILES, 66)],
                         ids=lambda v: getattr(v, "name", v))
def test_teacher_forced_logits_by_rows_and_widths(pkg, shape, rows):
    _check(pkg, shape, rows, Lp=5, T=3)


@pytest.mark.parametrize("rows", [2, 20])
@pytest.mark.parametrize("Lp", [30, 62, 126, 254, 638])
def test_new_position_at_tile_edges(pkg, Lp, rows):
    _check(pkg, ODD, rows, Lp, T=5)


# every row of the head is the same large vector: all logits of a position are equal, so large that their sums with the
# noise are rounded and tie
@pytest.mark.parametrize("shape,rows", [(NARROW, 3), (NARROW, 40), (VOCAB_TILES, 9)], ids=lambda v: getattr(v, "name", v))
def test_draws_from_large_logits(pkg, shape, rows):
    weights = dict(synth.model_weights(shape, 3))
    base = np.random.default_rng(1).standard_normal(shape.d_model).astype(np.float32) * 1e5
    weights["lm_head"] = np.ascontiguousarray(np.broadcast_to(synth.f32_to_bf16_bits(base), (shape.vocab, shape.d_model)))
    Lp, T = 4, 4
    rng = np.random.default_rng(rows)
    prompts = rng.integers(0, shape.vocab, size=(rows, Lp)).astype(np.int32)
    forced = rng.integers(0, shape.vocab, size=(rows, T)).astype(np.int32)
    uids = np.arange(rows, dtype=np.int64) * 64 + 3
    cfg = pkg.model_cfg(shape, max_prompts=rows, max_active=rows, max_seqs=rows, max_prompt_len=Lp, max_gen_len=T + 1,
                        max_k=2)
    with pkg.Handle(cfg, weights) as h:
        logits, sampled = h.teacher_force(prompts, forced, uids, sample_seed=9)
    assert np.abs(logits).min(axis=-1).max() > 1e5
    clear = sum(assert_drawn_by_the_rule(sampled[i, t], logits[i, t], 9, int(uids[i]), t) for i in range(rows) for t in range(T))
    assert clear >= rows * T // 2


def _check(pkg, shape, rows, Lp, T):
    weights = synth.model_weights(shape, 3)
    rng = np.random.default_rng(rows + shape.ffn)
    prompts = rng.integers(0, shape.vocab, size=(rows, Lp)).astype(np.int32)
    forced = rng.integers(0, shape.vocab, size=(rows, T)).astype(np.int32)
    uids = np.arange(rows, dtype=np.int64) * 64 + 3
    cfg = pkg.model_cfg(shape, max_prompts=rows, max_active=rows, max_seqs=rows, max_prompt_len=Lp, max_gen_len=T + 1,
                        max_k=2)
    with pkg.Handle(cfg, weights) as h:
        logits, sampled = h.teacher_force(prompts, forced, uids, sample_seed=9)
    want = o2.teacher_forced_logits_batch(o2.Weights(shape, weights), prompts, forced)
    err, rel = logit_errors(logits, want)
    assert err < LOGIT_MAX_ABS and rel < LOGIT_REL_L2, (err, rel)
    for i in range(rows):
        for t in range(T):
            tok, margin = o2.sample_token(logits[i, t], 9, int(uids[i]), t)
            if margin > 1e-4:
                assert sampled[i, t] == tok, (i, t)
