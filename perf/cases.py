"""What is timed: the calls a program that generates images makes, and how to compare their results.

Five kinds of case, all through the public Python entry points:

  generate   a prompt is pre-filled and `passes` iterations run (generate.generate): how an image starts
  decode     `passes` further iterations of an image that already has a long prefix (Context.step)
  verify     the verify-and-resample step alone (sjd_verify)
  attention  the window attention alone (sjd_attention)
  gemm       one projection alone (sjd_gemm)

Models are the repository's own workloads.  Their random weights are made decided: the embedding is N(0, 1),
the matrices that write into the residual stream are scaled by 1 / sqrt(2 * layers), and the output matrix is the
embedding shifted by one token, so that token t is followed by t + 1 with a probability that rounds to 1.  No token then
hangs on the last bit of a sum (two correct implementations agree on every token, for as many iterations as are
run), and an iteration fixes one token, as it does with plain random weights (about 1.03), so that a case's work
is known beforehand.  All the arithmetic of an iteration runs as with any other weights.
"""
import math

import torch

from paper_2410_01699_b200 import binding as B
from paper_2410_01699_b200.generate import generate
from paper_2410_01699_b200.inputs import WORKLOADS, make_weights

LOGIT = 64.0   # about 0.65 to 1 of it is the logit of the token that follows; all others are about N(0, (LOGIT / 64)^2) at d = 4096


def listed():
    gen = dict(kind="generate", guidance=0.0, init=B.SJD_INIT_RANDOM, ragged=False, paged=False, qk_norm=False)
    return [
        # the smallest model, fp32 storage: nothing but launches and latency
        dict(gen, name="tiny_f32", model="tiny", batch=1, window=16, prompt=16, passes=16),
        # a small bf16 model serving three prompts of different lengths
        dict(gen, name="small_bf16_ragged", model="small-bf16", batch=3, window=16, prompt=41, passes=16, ragged=True),
        # the headline use: one image of the 7B decoder from a text prompt
        dict(gen, name="7b_text", model="7b", batch=1, window=32, prompt=64, passes=12),
        # the same under classifier-free guidance (two streams), tokens copied from the grid row above
        dict(gen, name="7b_guided", model="7b", batch=1, window=16, prompt=45, passes=8, guidance=3.0,
             init=B.SJD_INIT_COPY_ABOVE),
        # a prompt that holds an image (1000 tokens and some text): pre-fill dominates
        dict(gen, name="7b_image_prompt", model="7b", batch=1, window=32, prompt=1063, passes=1),
        # eight images at a time from prompts of different lengths, paged cache
        dict(gen, name="7b_batch8", model="7b", batch=8, window=32, prompt=83, passes=3, ragged=True, paged=True),
        # grouped-query decoder with the large vocabulary and the widest window
        dict(gen, name="8b_gqa_w64", model="8b-gqa", batch=1, window=64, prompt=128, passes=6),
        # the end of a 7B image: every iteration reads about 2200 cached positions
        dict(kind="decode", name="7b_late", model="7b", batch=1, window=32, prompt=2161, passes=4),
        # verification of a serving batch, bf16 logits
        dict(kind="verify", name="verify_b32", batch=32, window=32, vocab=16384, dtype="bf16", top_k=2000, temperature=1.0),
        # verification of one window of fp32 logits over the 7B vocabulary, odd window
        dict(kind="verify", name="verify_b1_f32", batch=1, window=27, vocab=65536, dtype="f32", top_k=2000, temperature=0.9),
        # attention of eight late images
        dict(kind="attention", name="attention_b8", batch=8, window=32, prefix=3977, heads=32, kv_heads=32, head_dim=128),
        # the gate and up projections for a few hundred token rows
        dict(kind="gemm", name="gemm_m200", rows=200, n=22016, k=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("generate", "generate", "generate", "generate", "decode", "verify", "verify", "attention", "gemm"))
    if kind == "verify":
        dtype = rng.choice(("bf16", "bf16", "f32"))
        vocab = rng.choice((1024, 4096, 8192, 16384, 65536, _log_int(rng, 1000, 60000)))
        window = _log_int(rng, 4, 64)
        batch = max(1, min(_log_int(rng, 1, 32), (32 * 32 * 16384) // (window * vocab)))
        return dict(kind=kind, batch=batch, window=window, vocab=vocab, dtype=dtype, top_k=_log_int(rng, 8, vocab // 4),
                    temperature=round(rng.uniform(0.7, 1.3), 2))
    if kind == "attention":
        heads, kv_heads, hd = rng.choice(((32, 32, 128), (32, 8, 128), (8, 2, 64)))
        return dict(kind=kind, batch=rng.randint(1, 8), window=_log_int(rng, 4, 64), prefix=_log_int(rng, 60, 3977), heads=heads,
                    kv_heads=kv_heads, head_dim=hd)
    if kind == "gemm":
        return dict(kind=kind, rows=_log_int(rng, 8, 512), n=128 * rng.randint(8, 172), k=64 * rng.randint(8, 172))
    if kind == "decode":
        batch, window = rng.choice(((1, 16), (1, 32), (1, 64), (2, 32), (1, rng.randint(9, 63))))
        return dict(kind=kind, model=rng.choice(("7b", "7b", "8b-gqa")), batch=batch, window=window, prompt=rng.randint(300, 2161),
                    passes=rng.randint(2, 4))
    model = rng.choice(("tiny", "small-bf16", "small-bf16", "7b", "7b", "7b", "8b-gqa"))
    window = _log_int(rng, 4, 32 if model == "tiny" else 64)
    guidance = rng.choice((0.0, 0.0, 3.0))
    batch = _log_int(rng, 1, 8)
    batch = max(1, min(batch, (128 if model == "8b-gqa" else 256) // (window * (2 if guidance else 1))))
    prompt = _log_int(rng, 8, 200 if model in ("tiny", "small-bf16") else max(16, 1063 // (batch * (2 if guidance else 1))))
    return dict(kind="generate", model=model, batch=batch, window=window, prompt=prompt,
                passes=rng.randint(2, 16 if model in ("tiny", "small-bf16") else 4), guidance=guidance,
                init=rng.choice((B.SJD_INIT_RANDOM, B.SJD_INIT_RANDOM, B.SJD_INIT_COPY_ABOVE, B.SJD_INIT_COPY_LEFT,
                                 B.SJD_INIT_RESAMPLE_LEFT, B.SJD_INIT_RESAMPLE_ABOVE)),
                ragged=rng.random() < 0.4, paged=rng.random() < 0.3, qk_norm=rng.random() < 0.2)


# -------------------------------------------------------------------------------------------------- states
def _decided_weights(wl, seed, qk_norm):
    w = make_weights(wl.with_(weight_seed=seed), device="cuda", qk_norm=qk_norm)
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    emb = torch.randn(wl.vocab, wl.d_model, generator=gen, device="cuda")
    w["tok_emb"] = emb.to(w["tok_emb"].dtype)
    w["lm_head"] = (emb.roll(1, 0) * (LOGIT / wl.d_model)).to(w["lm_head"].dtype)
    for lw in w["layers"]:
        lw["wo"] *= (2 * wl.n_layers) ** -0.5
        lw["w_down"] *= (2 * wl.n_layers) ** -0.5
    return w


def _streams(case):
    return case["batch"] * (2 if case.get("guidance") else 1)


def _lens(case):
    """Prompt length of every stream; under guidance the two streams of an image share theirs."""
    p, n = case["prompt"], case["batch"]
    lens = [max(1, p - (i * p) // (2 * n)) if case.get("ragged") else p for i in range(n)]
    return [x for x in lens for _ in range(2)] if case.get("guidance") else lens


def _model_state(case, seed):
    wl = WORKLOADS[case["model"]]
    streams, lens = _streams(case), _lens(case)
    total = max(lens) + wl.n_generate
    ring = wl.grid_stride + case["window"] if case.get("init") == B.SJD_INIT_RESAMPLE_ABOVE else 0
    pages = sum(-(-(p + wl.n_generate) // 64) for p in lens) if case.get("paged") else 0
    ctx = B.Context(B.make_model_cfg(wl, streams, total, case["window"], ring, pages),
                    _decided_weights(wl, seed, case.get("qk_norm", False)))
    gen = torch.Generator(device="cuda").manual_seed(seed + 2)
    prompt = torch.randint(0, wl.vocab, (streams, max(lens)), generator=gen, device="cuda").to(torch.int32)
    if case.get("guidance"):   # both streams of an image end in the same token
        for i, n in enumerate(lens):
            prompt[i, n - 1] = prompt[i - i % 2, n - 1]
    sample = B.make_sample_cfg(temperature=wl.temperature, top_k=wl.top_k, seed=seed, window=case["window"],
                               init=case.get("init", B.SJD_INIT_RANDOM), grid_stride=wl.grid_stride,
                               n_generate=wl.n_generate, guidance=case.get("guidance", 0.0))
    return dict(case=case, ctx=ctx, prompt=prompt, sample=sample, lens=lens if case.get("ragged") else None)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "generate":
        return _model_state(case, seed)
    if kind == "decode":
        s = _model_state(case, seed)
        s["ctx"].prefill(s["prompt"], s["sample"])
        s["out"] = B.StepOut(case["batch"], case["window"])
        return s
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def randn(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    if kind == "verify":
        # the distribution of inputs.make_verify_case: N(0, 3^2) with 5 % of the entries raised by 6, the previous
        # rows are those plus N(0, 1), drafts drawn from the previous rows' top-k by the Gumbel-max trick; a quarter
        # each of the slots is freshly initialised at random or copied
        b, w, v = case["batch"], case["window"], case["vocab"]
        dt = {"bf16": torch.bfloat16, "f32": torch.float32}[case["dtype"]]
        cur = 3.0 * randn(b, w, v)
        cur += 6.0 * (torch.rand(b, w, v, generator=gen, device="cuda") < 0.05)
        prev = (cur + randn(b, w, v)).to(dt)
        cur = cur.to(dt)
        scaled = prev.float() / case["temperature"]
        kth = scaled.topk(min(case["top_k"], v), dim=-1).values[..., -1:]
        gumbel = -torch.log(-torch.log(torch.rand(b, w, v, generator=gen, device="cuda").clamp(1e-7, 1 - 1e-7)))
        draft = torch.where(scaled >= kth, scaled + gumbel, torch.full_like(scaled, -math.inf)).argmax(-1)
        q_kind = torch.tensor([B.SJD_Q_ROW, B.SJD_Q_ROW, B.SJD_Q_UNIFORM, B.SJD_Q_ONEHOT], device="cuda")[
            torch.randint(0, 4, (b, w), generator=gen, device="cuda")]
        draft = torch.where(q_kind == B.SJD_Q_UNIFORM, torch.randint(0, v, (b, w), generator=gen, device="cuda"), draft)
        draft = torch.where(q_kind == B.SJD_Q_ONEHOT, cur.float().argmax(-1), draft)
        base = torch.randint(16, 4096, (b,), generator=gen, device="cuda")
        return dict(case=case, cur=cur, prev=prev, draft=draft.to(torch.int32), q_kind=q_kind.to(torch.int32),
                    base=base.to(torch.int32), out=B.StepOut(b, w),
                    sample=B.make_sample_cfg(temperature=case["temperature"], top_k=case["top_k"], seed=seed, window=w),
                    ws=torch.empty(B.sjd_verify_workspace_bytes(b, w), dtype=torch.uint8, device="cuda"))
    if kind == "attention":
        b, w, n, hd = case["batch"], case["window"], case["prefix"], case["head_dim"]
        kv = torch.stack([randn(2, case["kv_heads"], n + w, hd).to(torch.bfloat16) for _ in range(b)])
        pos = (n - 1 + torch.arange(w, dtype=torch.int32, device="cuda")).repeat(b).contiguous()
        return dict(case=case, q=randn(b * w, case["heads"], hd), kv=kv, pos=pos)
    return dict(case=case, x=randn(case["rows"], case["k"]), w=(0.02 * randn(case["n"], case["k"])).to(torch.bfloat16))


# -------------------------------------------------------------------------------------------------- passes
def _all_of(out):
    return {n: getattr(out, n) for n in ("n_accepted", "n_committed", "committed", "draft", "q_kind", "q_draft", "total_committed",
                                         "flags")}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "generate":
        tokens, counts, _ = generate(state["ctx"], state["prompt"], state["sample"], prompt_lens=state["lens"],
                                     max_steps=case["passes"])
        return {"tokens": tokens, "counts": counts, "logits": state["ctx"].peek_logits()}
    if kind == "decode":
        for _ in range(case["passes"]):
            state["ctx"].step(state["out"])
        return {"logits": state["ctx"].peek_logits(), **_all_of(state["out"])}
    if kind == "verify":
        B.sjd_verify(state["cur"], state["prev"], state["draft"], state["q_kind"], state["base"], state["sample"], 7, state["out"],
                     ws=state["ws"])
        return _all_of(state["out"])
    if kind == "attention":
        return B.sjd_attention(state["q"], state["kv"], state["pos"], case["window"], case["kv_heads"])[0]
    return B.sjd_gemm(state["x"], state["w"])[0]


# -------------------------------------------------------------------------------------------------- bounds
def work(case):
    kind = case["kind"]
    if kind == "verify":
        n = case["batch"] * case["window"] * case["vocab"]
        return {"bytes": 2 * n * (2 if case["dtype"] == "bf16" else 4), "flops": 0}
    if kind == "attention":
        b, w, n, hd = case["batch"], case["window"], case["prefix"], case["head_dim"]
        return {"bytes": b * 2 * case["kv_heads"] * (n + w) * hd * 2 + 2 * b * w * case["heads"] * hd * 4,
                "flops": 4 * b * w * case["heads"] * (n + w / 2) * hd}
    if kind == "gemm":
        m, n, k = case["rows"], case["n"], case["k"]
        return {"bytes": 2 * n * k + 4 * m * (n + k), "flops": 2 * m * n * k}
    wl = WORKLOADS[case["model"]]
    es = 4 if wl.dtype == "f32" else 2
    lens = _lens(case)
    kv_row = wl.n_layers * 2 * wl.n_kv_heads * wl.head_dim * es   # cache bytes of one position
    head = wl.vocab * wl.d_model * es
    mats = wl.step_weight_bytes() / es
    per_key = 4 * wl.n_layers * wl.n_heads * wl.head_dim           # attention flops of one query and one key
    nbytes = flops = 0.0
    if kind == "generate":   # the prompt goes through the layers once
        rows = sum(n - 1 for n in lens)
        nbytes += (wl.step_weight_bytes() - head if rows else 0) + rows * kv_row
        flops += 2 * (mats - head / es) * rows + per_key * sum(n * n / 2 for n in lens)
    w = case["window"]
    for i in range(case["passes"]):   # one token fixed by each pass
        keys = sum(n + i + w for n in lens)
        nbytes += wl.step_weight_bytes() + keys * kv_row + len(lens) * (w + 1) * wl.vocab * es
        flops += 2 * mats * len(lens) * w + per_key * keys * w
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the difference measured between two correct versions: the projections, the attention split and
    the generic products with their sums in another order for whole models, double precision for single kernels."""
    kind = case["kind"]
    if kind == "verify":      # fp32 weights; a draw by inverse CDF may land on the other side of a token boundary
        return {"rel": 1e-5, "max": 1e-3, "differ": 0.002}
    if kind in ("attention", "gemm"):   # 5.8e-6 and 5.1e-6 against double precision, largest 3.1e-5 and 2.2e-5
        return {"rel": 2.4e-5, "max": 1.2e-4}
    if WORKLOADS[case["model"]].dtype == "f32":   # 3.0e-7, largest 1.5e-6, with the inner sums in another order
        return {"rel": 3e-6, "max": 2e-5}
    return {"rel": 7e-3, "max": 0.04}   # bf16 cache and logits: 1.8e-3, largest 7.8e-3 (one bf16 step), tokens identical
