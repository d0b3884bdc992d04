"""Shared helpers of the GPU parity tests (inputs from synth, expectations from oracle/)."""
import numpy as np

from oracle import decode as o2

LOGIT_MAX_ABS = 3e-2   # per-step logits under teacher forcing (the stated parity tolerance)
LOGIT_REL_L2 = 1e-2


def handle_cfg(w, pkg, max_seqs=None, max_prompts=None):
    return pkg.model_cfg(w.model, max_prompts=max_prompts or w.n_prompts, max_active=w.target_B,
                         max_seqs=max_seqs or w.target_B * w.n0, max_prompt_len=w.prompt_len,
                         max_gen_len=w.lengths.max_len, max_k=w.k)


def logit_errors(got, want):
    err = float(np.abs(got - want).max())
    rel = float(np.linalg.norm(got - want) / np.linalg.norm(want))
    return err, rel


def assert_drawn_by_the_rule(tok, logits_row, sample_seed, uid, t):
    """tok is the first maximum of fp32 logit + noise.  The device's logarithms may be an ulp or two off the host's (noise
    below 17: 1e-5 is several), which can move a sum across a rounding: any token that could then be the maximum passes.
    Returns whether there was no such doubt (a single answer)."""
    z = logits_row.astype(np.float64) + o2.gumbel_noise(sample_seed, uid, t, logits_row.shape[-1]).astype(np.float64)
    lo, hi = (z - 1e-5).astype(np.float32), (z + 1e-5).astype(np.float32)
    could = np.flatnonzero(hi >= lo.max())
    assert tok in could, (tok, could)
    if not np.array_equal(lo[could], hi[could]):
        return False
    assert tok == could[0], (tok, could)
    return True
