"""Performance cases: the work a user of the rollout-collection library has it do, through its public entry points.

Kinds of cases:

  gemm     one projection of up to 128 activation rows (`gemm_bf16`, or `gemm_bf16_static` for callers that cannot
           allocate device memory)
  attn     grouped-query attention of single query rows over their own ragged KV histories (`attention_decode`)
  sample   the temperature-1 draw from given logits (`sample`)
  force    prefill of the prompts, then teacher-forced decode steps whose logits come back (`sara_teacher_force` on
           device buffers, as a policy's log-probabilities are recomputed): short prompts with many steps are the decode
           step, long prompts with one step the prefill.  One or a few decoder layers between the embedding and the
           head stand for the layers and blocks, the full depth for the whole model
  collect  one rollout-collection step with the policy (`Handle.collect_step`): controller, prefill, decode, sampling
  control  the controller alone, on a handle without a model

Shapes are the repository's workloads (1.5B- and 3B-shaped policies, the tiny policy, the controller sweep).
"""
import ctypes
import math

import numpy as np
import torch

import paper_2607_26253_gb300 as sara

SHAPES = {
    "tiny": dict(d=128, heads=4, kv=2, hd=32, ffn=512, vocab=512),
    "1.5b": dict(d=1536, heads=12, kv=2, hd=128, ffn=8960, vocab=151936),
    "3b": dict(d=2048, heads=16, kv=2, hd=128, ffn=11008, vocab=151936),
}
DEPTH = {"tiny": 2, "1.5b": 28, "3b": 36}
# (Nout, K) of the two policies' projections: q|k|v, output, gate|up, down, head
GEMMS = [(2048, 1536), (1536, 1536), (17920, 1536), (1536, 8960), (151936, 1536),
         (2560, 2048), (2048, 2048), (22016, 2048), (2048, 11008), (151936, 2048)]
ATTN_HEADS = [(12, 2, 128), (16, 2, 128), (8, 2, 128), (8, 8, 64), (4, 2, 32)]  # query heads, KV heads, head dim
FEW_TOKENS = 400  # below this many draws one near-tie is too large a share of them to compare tokens
ROPE_THETA, RMS_EPS = 1.0e6, 1.0e-6


def listed():
    return [
        # the smallest call: one row through the q|k|v projection, where launch and latency count
        {"name": "gemm 1 row qkv", "kind": "gemm", "rows": 1, "n": 2048, "k": 1536, "static": False},
        # a full 64-row batch through the vocabulary head: the largest weight, bound by reading it
        {"name": "gemm 64 rows head", "kind": "gemm", "rows": 64, "n": 151936, "k": 1536, "static": False},
        # the allocation-free entry point, an odd row count through the widest reduction
        {"name": "gemm 33 rows down static", "kind": "gemm", "rows": 33, "n": 2048, "k": 11008, "static": True},
        # attention of a mid-step batch over ragged contexts
        {"name": "attention 26 rows", "kind": "attn", "rows": 26, "heads": 12, "kv": 2, "hd": 128, "ctx": 758},
        # sampling from a batch's logits over the whole vocabulary
        {"name": "sample 64 rows", "kind": "sample", "rows": 64, "vocab": 151936},
        # one decoder layer, a single live rollout: the long tail of every round
        {"name": "layer decode 1 row", "kind": "force", "shape": "1.5b", "layers": 1, "rows": 1, "prompt": 33,
         "steps": 24},
        # two layers of the wider policy at more than 64 live rows: the start of a round
        {"name": "layers decode 80 rows 3b", "kind": "force", "shape": "3b", "layers": 2, "rows": 80, "prompt": 17,
         "steps": 12},
        # fresh prompts of a round: two layers over 64 prompts of 256 tokens, one decode step
        {"name": "prefill 64 x 256", "kind": "force", "shape": "1.5b", "layers": 2, "rows": 64, "prompt": 256,
         "steps": 1},
        # the whole 1.5B-shaped model at its mean number of live rows
        {"name": "model decode 26 rows", "kind": "force", "shape": "1.5b", "layers": 28, "rows": 26, "prompt": 40,
         "steps": 32},
        # a whole collection step of the tiny policy: many short decode steps, controller between them
        {"name": "collect tiny", "kind": "collect", "shape": "tiny", "layers": 2, "pool": 64, "target": 16, "k": 8,
         "n0": 2, "budget": 128, "prompt": 32, "median": 18, "cap": 32, "schedule": 0},
        # a whole collection step of the 1.5B-shaped policy, its lengths scaled down to keep a pass short
        {"name": "collect 1.5b", "kind": "collect", "shape": "1.5b", "layers": 28, "pool": 48, "target": 16, "k": 8,
         "n0": 2, "budget": 96, "prompt": 64, "median": 32, "cap": 128, "schedule": 0},
        # the controller over a large pool, without a policy
        {"name": "controller 65536 prompts", "kind": "control", "pool": 65536, "target": 8192, "k": 8, "n0": 2,
         "budget": 262144, "schedule": 0},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["gemm", "attn", "sample", "force", "force", "force", "force", "collect", "control"])
    if kind == "gemm":
        n, k = rng.choice(GEMMS) if rng.random() < 0.5 else (128 * _log_int(rng, 1, 800), 64 * _log_int(rng, 1, 172))
        while n * k > 151936 * 2048:
            n = max(128, n // 256 * 128)
        return {"kind": kind, "rows": _log_int(rng, 1, 128), "n": n, "k": k, "static": rng.random() < 0.3}
    if kind == "attn":
        heads, kv, hd = rng.choice(ATTN_HEADS)
        return {"kind": kind, "rows": _log_int(rng, 1, 128), "heads": heads, "kv": kv, "hd": hd,
                "ctx": _log_int(rng, 16, 4096)}
    if kind == "sample":
        return {"kind": kind, "rows": _log_int(rng, 1, 128), "vocab": rng.choice([151936, 151936, 512, 32000 + rng.randrange(999)])}
    if kind == "force":
        shape = rng.choice(["1.5b", "1.5b", "3b", "tiny"])
        rows = _log_int(rng, 1, 128)
        if rng.random() < 0.5:  # decode: many steps after a short prompt
            steps = max(2, min(_log_int(rng, 4, 64), 2048 // rows))
            prompt = _log_int(rng, 2, 96)
        else:                   # prefill: the prompts' tokens, at most 32,768 of them, and a step or two
            steps = rng.randrange(1, 3)
            prompt = min(_log_int(rng, 32, 2048), max(2, 32768 // rows))
        return {"kind": kind, "shape": shape, "layers": rng.randrange(1, 4), "rows": rows, "prompt": prompt,
                "steps": steps}
    if kind == "collect":
        target, k = _log_int(rng, 2, 32), rng.choice([4, 8, 8, 16])
        median = _log_int(rng, 6, 24)
        return {"kind": kind, "shape": rng.choice(["tiny", "1.5b"]), "layers": rng.randrange(1, 4), "pool": 3 * target,
                "target": target, "k": k, "n0": rng.choice([1, 2, 3]), "budget": target * k * 3 // 4,
                "prompt": _log_int(rng, 8, 128), "median": median, "cap": 4 * median, "schedule": rng.choice([0, 0, 1, 2])}
    target = _log_int(rng, 256, 8192)
    return {"kind": kind, "pool": 8 * target, "target": target, "k": rng.choice([4, 8, 16]), "n0": rng.choice([1, 2, 3]),
            "budget": 8 * target * rng.choice([1, 2, 4]), "schedule": 0}


# ------------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _randn(g, shape, dtype, std=1.0):
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype).mul_(std)


def _randint(g, hi, shape, dtype=torch.int32):
    return torch.randint(0, hi, shape, generator=g, device="cuda", dtype=dtype)


class _Shape:
    def __init__(self, name, layers):
        s = SHAPES[name]
        self.layers, self.d_model, self.n_heads, self.n_kv_heads = layers, s["d"], s["heads"], s["kv"]
        self.head_dim, self.ffn, self.vocab = s["hd"], s["ffn"], s["vocab"]
        self.rope_theta, self.rms_eps = ROPE_THETA, RMS_EPS


def _weights(case, g):
    """A random policy on the GPU, drawn tensor by tensor: N(0, 0.02) projections, norm weights around 1."""
    s = SHAPES[case["shape"]]
    d, q, kv, f, v = s["d"], s["heads"] * s["hd"], s["kv"] * s["hd"], s["ffn"], s["vocab"]
    w = lambda *shape: _randn(g, shape, torch.bfloat16, 0.02)  # noqa: E731
    norm = lambda: _randn(g, (d,), torch.bfloat16, 0.1).add_(1.0)  # noqa: E731
    out = {"embed": w(v, d), "final_norm": norm(), "lm_head": w(v, d), "layers": []}
    for _ in range(case["layers"]):
        out["layers"].append({"attn_norm": norm(), "wq": w(q, d), "wk": w(kv, d), "wv": w(kv, d), "wo": w(d, q),
                              "mlp_norm": norm(), "wgate": w(f, d), "wup": w(f, d), "wdown": w(d, f)})
    return out


def _force_inputs(case, seed):
    g = _gen(seed)
    w = _weights(case, g)
    v, n = SHAPES[case["shape"]]["vocab"], case["rows"]
    return w, _randint(g, v, (n, case["prompt"])), _randint(g, v, (n, case["steps"]))


def _latent_thresholds(rng, n):
    """Success rates of the prompts: 35 % never, 25 % always, else Beta(2, 2); as floor(p * 2^32)."""
    comp, b = rng.random(n), np.median(rng.random((n, 3)), axis=1)
    p = np.where(comp < 0.35, 0.0, np.where(comp < 0.60, 1.0, b))
    t = np.floor(p * 4294967296.0).astype(np.uint64)
    t[p >= 1.0] = np.uint64(1 << 32)
    return t


def _attn_inputs(case, seed):
    g, rng = _gen(seed), np.random.default_rng(seed)
    b, hd = case["rows"], case["hd"]
    ctx = np.clip(np.rint(case["ctx"] * np.exp(0.5 * rng.standard_normal(b))), 1, 3 * case["ctx"]).astype(np.int32)
    cap = int(ctx.max())
    q = _randn(g, (b, case["heads"], hd), torch.float16)
    kv = _randn(g, (b, 2, case["kv"], cap, hd), torch.float16)
    return q, kv, ctx, cap


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "gemm":
        g = _gen(seed)
        r, n, k = case["rows"], case["n"], case["k"]
        st["x"] = _randn(g, (r, k), torch.bfloat16)
        st["w"] = _randn(g, (n, k), torch.bfloat16, 0.02)
        if not case["static"]:
            st["ws"] = torch.zeros(sara.load().sara_gemm_workspace_bytes(r, n, k), dtype=torch.uint8, device="cuda")
    elif kind == "attn":
        st["q"], st["kv"], ctx, st["cap"] = _attn_inputs(case, seed)
        st["ctx"] = torch.from_numpy(ctx).cuda()
    elif kind == "sample":
        g = _gen(seed)
        r = case["rows"]
        st["logits"] = _randn(g, (r, case["vocab"]), torch.float32, 2.0)
        st["uid"] = _randint(g, 1 << 20, (r,), torch.int64)
        st["t"] = _randint(g, 4096, (r,))
        st["seed"] = seed
    elif kind == "force":
        w, st["prompts"], st["forced"] = _force_inputs(case, seed)
        n, steps = case["rows"], case["steps"]
        cfg = sara.model_cfg(_Shape(case["shape"], case["layers"]), max_prompts=n, max_active=n, max_seqs=n,
                             max_prompt_len=case["prompt"], max_gen_len=steps + 1, max_k=2)
        st["handle"] = sara.Handle(cfg, w)
        st["uid"] = torch.arange(n, dtype=torch.int64, device="cuda") * 64 + 1
        st["logits"] = torch.empty((n, steps, SHAPES[case["shape"]]["vocab"]), dtype=torch.float32, device="cuda")
        st["tokens"] = torch.empty((n, steps), dtype=torch.int32, device="cuda")
        st["seed"] = seed
    else:
        rng = np.random.default_rng(seed)
        P, k = case["pool"], case["k"]
        st["thresholds"] = _latent_thresholds(rng, P)
        st["seed"] = seed
        if kind == "collect":
            w = _weights(case, _gen(seed))
            x = np.rint(case["median"] * np.exp(0.5 * rng.standard_normal((P, k))))
            st["lengths"] = np.clip(x, 1, case["cap"]).astype(np.int32)
            st["tokens"] = rng.integers(0, SHAPES[case["shape"]]["vocab"], (P, case["prompt"])).astype(np.int32)
            cfg = sara.model_cfg(_Shape(case["shape"], case["layers"]), max_prompts=P, max_active=case["target"],
                                 max_seqs=min(128, case["target"] * max(case["n0"], 2)), max_prompt_len=case["prompt"],
                                 max_gen_len=case["cap"], max_k=k)
            st["handle"] = sara.Handle(cfg, w)
        else:
            st["lengths"], st["tokens"] = np.ones((P, k), np.int32), None
            cfg = sara.model_cfg(None, max_prompts=P, max_active=case["target"], max_seqs=1, max_prompt_len=1,
                                 max_gen_len=1, max_k=k)
            st["handle"] = sara.Handle(cfg)
    return st


# ------------------------------------------------------------------------------------------------ one pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "gemm":
        if case["static"]:
            return sara.gemm_bf16_static(state["x"], state["w"])
        return sara.gemm_bf16(state["x"], state["w"], workspace=state["ws"])
    if kind == "attn":
        return sara.attention_decode(state["q"], state["kv"], state["ctx"], case["kv"], state["cap"],
                                     max_ctx=state["cap"])
    if kind == "sample":
        return sara.sample(state["logits"], state["uid"], state["t"], state["seed"])
    if kind == "force":
        h, p = state["handle"], lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
        rc = sara.load().sara_teacher_force(h._h, case["rows"], case["prompt"], p(state["prompts"]), case["steps"],
                                            p(state["forced"]), p(state["uid"]), state["seed"], p(state["logits"]),
                                            p(state["tokens"]), 1)
        if rc != sara.SARA_OK:
            raise sara.SaraError(rc, sara.load().sara_last_error(h._h).decode())
        out = {"logits": state["logits"]}
        if case["rows"] * case["steps"] >= FEW_TOKENS:
            out["tokens"] = state["tokens"]
        return out
    # The outcomes of every prompt and the step's counters.  They do not depend on the policy's tokens, whose draws
    # may part for good after one near-tie; the same kernels' logits and draws come back in the "force" cases.
    o = state["handle"].collect_step(thresholds=state["thresholds"], lengths=state["lengths"], tokens=state["tokens"],
                                     N=case["budget"], k=case["k"], n0=case["n0"], tau=0.45, target_B=case["target"],
                                     reward_seed=state["seed"], sample_seed=state["seed"], schedule=case["schedule"])
    return {"status": o.status, "n": o.n, "s": o.s, "round": o.decided_round, "counters": o.counters}


# ------------------------------------------------------------------------------------------------ necessary work
def _layer_params(s):
    q, kv = s["heads"] * s["hd"], s["kv"] * s["hd"]
    return s["d"] * (q + 2 * kv) + q * s["d"] + 3 * s["d"] * s["ffn"]


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        r, n, k = case["rows"], case["n"], case["k"]
        return {"bytes": 2 * (r * k + n * k) + 4 * r * n, "flops": 2 * r * n * k}
    if kind == "attn":
        pos = case["rows"] * case["ctx"] * 1.13  # the mean of the ragged contexts
        return {"bytes": pos * case["kv"] * case["hd"] * 4 + case["rows"] * case["heads"] * case["hd"] * 4,
                "flops": pos * case["heads"] * case["hd"] * 4}
    if kind == "sample":
        return {"bytes": case["rows"] * case["vocab"] * 4, "flops": case["rows"] * case["vocab"] * 20}
    if kind == "control":
        # thresholds and lengths in, outcomes out, once per prompt
        return {"bytes": case["pool"] * (8 + 4 * case["k"] + 5), "flops": 0}
    s = SHAPES[case["shape"]]
    layer, head, kvtok = _layer_params(s), s["vocab"] * s["d"], case["layers"] * s["kv"] * s["hd"] * 4
    params = case["layers"] * layer
    if kind == "force":
        n, lp, t = case["rows"], case["prompt"], case["steps"]
        ctx = t * (lp - 1) + t * (t + 1) // 2  # positions read by one row's decode steps
        pre = n * (lp - 1)
        att = 4 * case["layers"] * s["heads"] * s["hd"]  # flops per query and position
        return {"bytes": 2 * params * (1 + t) + 2 * head * t + n * ctx * kvtok + (pre + n * t) * kvtok
                         + 2 * s["d"] * (pre + n * t) + 4 * n * t * s["vocab"],
                "flops": 2 * params * (pre + n * t) + 2 * head * n * t + att * n * (ctx + (lp - 1) * lp // 2)}
    # collect: at least this many decode steps, the batch as full as the working set allows
    rows = case["target"] * case["n0"]
    toks = case["budget"] * case["median"] * 1.1
    steps = toks / rows
    pre = case["target"] * (case["prompt"] - 1)
    return {"bytes": (2 * params + 2 * head) * steps + 2 * params + toks * kvtok * (case["prompt"] + case["median"] / 2),
            "flops": 2 * (params + head) * toks + 2 * params * pre}


# ------------------------------------------------------------------------------------------------ comparison
def tolerance(case):
    kind = case["kind"]
    if kind in ("collect", "control"):
        return "exact"
    if kind == "gemm":
        return {"rel": 1.2e-5, "max": 1.2e-4}   # 32-bit sums of exact products: 2.9e-6 at K = 11,008
    if kind == "attn":
        return {"rel": 1e-2, "max": 5e-2}   # results in bf16
    if kind == "sample":
        return {"rel": 0.0, "differ": 0.01}
    # activations as 16-bit-mantissa pairs, q, K, V in fp16, 32-bit sums; the depth adds up
    return {"rel": 4e-3, "max": 4e-2, "differ": 0.01}


# ------------------------------------------------------------------------------------------------ 64-bit results
def _rms(x, w):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + RMS_EPS) * w.double()


def _rotate(x, cos, sin):
    a, b = x.chunk(2, dim=-1)
    return torch.cat([a * cos - b * sin, b * cos + a * sin], dim=-1)


def _exact_logits(case, seed):
    w, prompts, forced = _force_inputs(case, seed)
    s = SHAPES[case["shape"]]
    toks = torch.cat([prompts, forced[:, :-1]], dim=1).long()
    n, L = toks.shape
    hd, H, KV = s["hd"], s["heads"], s["kv"]
    x = w["embed"][toks].double()
    inv = ROPE_THETA ** (-torch.arange(0, hd, 2, dtype=torch.float64, device="cuda") / hd)
    ang = torch.arange(L, dtype=torch.float64, device="cuda")[:, None] * inv[None, :]
    cos, sin = ang.cos(), ang.sin()
    mask = torch.full((L, L), -math.inf, dtype=torch.float64, device="cuda").triu(1)
    lin = lambda a, b: a @ b.double().t()  # noqa: E731
    for lw in w["layers"]:
        y = _rms(x, lw["attn_norm"])
        q = _rotate(lin(y, lw["wq"]).view(n, L, H, hd).transpose(1, 2), cos, sin)
        k = _rotate(lin(y, lw["wk"]).view(n, L, KV, hd).transpose(1, 2), cos, sin).repeat_interleave(H // KV, dim=1)
        v = lin(y, lw["wv"]).view(n, L, KV, hd).transpose(1, 2).repeat_interleave(H // KV, dim=1)
        o = torch.empty_like(q)
        for i in range(n):  # one sequence at a time: the scores stay small
            o[i] = torch.softmax(q[i] @ k[i].transpose(-1, -2) / math.sqrt(hd) + mask, dim=-1) @ v[i]
        x = x + lin(o.transpose(1, 2).reshape(n, L, H * hd), lw["wo"])
        y = _rms(x, lw["mlp_norm"])
        x = x + lin(torch.nn.functional.silu(lin(y, lw["wgate"])) * lin(y, lw["wup"]), lw["wdown"])
    return lin(_rms(x[:, case["prompt"] - 1:], w["final_norm"]), w["lm_head"])


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        g = _gen(seed)
        x = _randn(g, (case["rows"], case["k"]), torch.bfloat16)
        w = _randn(g, (case["n"], case["k"]), torch.bfloat16, 0.02)
        return x.double() @ w.double().t()
    if kind == "attn":
        q, kv, ctx, _ = _attn_inputs(case, seed)
        G = case["heads"] // case["kv"]
        out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
        for i, c in enumerate(ctx.tolist()):
            k, v = (kv[i, j, :, :c].double().repeat_interleave(G, dim=0) for j in (0, 1))
            p = torch.softmax((k @ q[i].double()[:, :, None])[..., 0] / math.sqrt(case["hd"]), dim=-1)
            out[i] = (p[:, None, :] @ v)[:, 0]
        return out
    if kind == "force":
        s = SHAPES[case["shape"]]
        tokens = case["rows"] * (case["prompt"] + case["steps"])
        flops = 2 * case["layers"] * _layer_params(s) * tokens + 2 * s["vocab"] * s["d"] * case["rows"] * case["steps"]
        if flops > 8e12:  # too long in 64 bits
            return None
        out = {"logits": _exact_logits(case, seed)}
        if case["rows"] * case["steps"] >= FEW_TOKENS:
            out["tokens"] = None
        return out
    return None
