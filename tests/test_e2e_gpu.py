"""GPU parity of sjd_init / sjd_prefill / sjd_step (through the C-ABI) against the CPU checker in
lock-step: before every step the checker holds the library's state; it recomputes the logits
itself (compared within the storage-dtype tolerance) and re-takes every decision of the step from
the library's stored logits (compared exactly, near-ties flagged)."""
import numpy as np
import pytest
import torch

from oracle.sjd import (INIT_COPY_ABOVE, INIT_COPY_LEFT, INIT_RANDOM, INIT_RESAMPLE_ABOVE, INIT_RESAMPLE_LEFT,
                        SampleCfg)
from paper_2410_01699_b200 import binding as B
from paper_2410_01699_b200.inputs import WORKLOADS, make_prompt, make_weights
from tests.parity_util import LockStepSequence, run_in_threads

pytestmark = pytest.mark.gpu

LOGIT_TOL = {"f32": 1e-4, "bf16": 2e-2}


def run_lockstep(wl, batch=1, max_steps=None, init=INIT_RANDOM, check_logits_every=1, gain_jitter=0.1, window=None,
                 n_generate=None, seq_base=0, top_k=None, also_plain_cache=False, schedule=0, qk_norm=False):
    window = window or wl.window
    n_generate = wl.n_generate if n_generate is None else n_generate
    top_k = top_k or wl.top_k
    weights = make_weights(wl, gain_jitter=gain_jitter, qk_norm=qk_norm)
    prompt = make_prompt(wl, batch)
    cfg = B.make_model_cfg(wl, max_batch=batch, max_seq=wl.prompt_len + n_generate + 8, max_window=window,
                           max_ring=wl.grid_stride + window if init == INIT_RESAMPLE_ABOVE else 0)
    ctx = B.Context(cfg, B.weights_to_device(weights))
    sample = B.make_sample_cfg(temperature=wl.temperature, top_k=top_k, seed=wl.philox_seed, window=window,
                               init=init, grid_stride=wl.grid_stride, n_generate=n_generate, seq_base=seq_base,
                               schedule=schedule)
    scfg = SampleCfg(temperature=wl.temperature, top_k=top_k, seed=wl.philox_seed, window=window, init=init,
                     grid_stride=wl.grid_stride, n_generate=n_generate, logits_dtype=wl.dtype, schedule=schedule)
    ctx.prefill(torch.from_numpy(prompt).cuda(), sample)
    out = B.StepOut(batch, window)
    ctx.get_window(out)
    h = out.host()
    seqs = [LockStepSequence(wl, weights, prompt[b], scfg, seq_base + b, LOGIT_TOL[wl.dtype], also_plain_cache)
            for b in range(batch)]
    for b, s in enumerate(seqs):
        s.check_window(h["draft"][b], h["q_kind"][b], h["q_draft"][b], h["total_committed"][b])
    steps = 0
    total = wl.prompt_len + n_generate
    committed = [list(prompt[b]) for b in range(batch)]
    while any(s.st.n < total for s in seqs):
        ctx.step(out)
        logits = ctx.peek_logits().to(torch.float64).cpu().numpy()
        h = out.host()
        for b, s in enumerate(seqs):
            ob = {k: v[b] for k, v in h.items()}
            s.step(logits[b], ob, check_logits=(steps % check_logits_every == 0))
            committed[b] += [int(t) for t in ob["committed"][:int(ob["n_committed"])]]
            assert committed[b] == s.st.committed
        steps += 1
        assert steps <= n_generate, "more forward passes than tokens"
        if max_steps and steps >= max_steps:
            break
    assert ctx.device_status() == B.SJD_OK
    # the sequences as the library hands them out (sjd_get_tokens): prompt + every token fixed so far
    tokens, counts = ctx.get_tokens()
    tokens, counts = tokens.cpu().numpy(), counts.cpu().numpy()
    for b, s in enumerate(seqs):
        assert int(counts[b]) == s.st.n
        assert [int(t) for t in tokens[b][:s.st.n]] == s.st.committed
    return ctx, seqs, steps, out


@pytest.mark.parametrize("name,batch,guidance", [("tiny", 3, 0.0), ("small-bf16", 2, 0.0), ("small-bf16", 4, 3.0)])
def test_generate_reproduces_the_lockstep_run(name, batch, guidance):
    """generate() (iterations enqueued without the host looking at them, DONE flags read every few
    iterations, sjd_get_tokens at the end) yields exactly the sequences of the run that was checked against
    the oracle step by step: the kernels are deterministic, so a second context must repeat them."""
    from paper_2410_01699_b200.generate import generate
    wl = WORKLOADS[name]
    n_generate = 45
    if guidance:
        checked, _ = run_lockstep_guided(wl, images=batch // 2, guidance=guidance, n_generate=n_generate)
    else:
        _, checked, _, _ = run_lockstep(wl, batch=batch, n_generate=n_generate)
    weights = make_weights(wl, gain_jitter=0.1)
    ctx = B.Context(B.make_model_cfg(wl, batch, wl.prompt_len + n_generate + 8, wl.window), B.weights_to_device(weights))
    sample = B.make_sample_cfg(temperature=wl.temperature, top_k=wl.top_k, seed=wl.philox_seed, window=wl.window,
                               init=INIT_RANDOM, grid_stride=wl.grid_stride, n_generate=n_generate, guidance=guidance)
    tokens, counts, steps = generate(ctx, torch.from_numpy(make_prompt(wl, batch)).cuda(), sample, check_every=5)
    tokens, counts = tokens.cpu().numpy(), counts.cpu().numpy()
    assert steps <= n_generate and len(checked) == len(counts)
    for i, s in enumerate(checked):
        assert int(counts[i]) == wl.prompt_len + n_generate
        assert [int(t) for t in tokens[i][:counts[i]]] == s.st.committed


@pytest.mark.parametrize("name,init,kv_pages", [("tiny", INIT_RESAMPLE_ABOVE, 0), ("small-bf16", INIT_RESAMPLE_ABOVE, 6),
                                                ("small-bf16", INIT_COPY_LEFT, 0)])
def test_second_prefill_starts_clean(name, init, kv_pages):
    """A context that has generated one batch and is pre-filled again (other prompts, other lengths of batch)
    yields what a fresh context yields: no window state, retained row, cache row or page of the first run
    leaks into the second."""
    from paper_2410_01699_b200.generate import generate
    wl = WORKLOADS[name]
    n_generate = 40
    weights = B.weights_to_device(make_weights(wl, gain_jitter=0.1))
    ring = wl.grid_stride + wl.window if init == INIT_RESAMPLE_ABOVE else 0

    def ctx():
        return B.Context(B.make_model_cfg(wl, 3, wl.prompt_len + n_generate + 8, wl.window, max_ring=ring,
                                          kv_pages=kv_pages), weights)

    def sample(seed):
        return B.make_sample_cfg(temperature=wl.temperature, top_k=wl.top_k, seed=seed, window=wl.window, init=init,
                                 grid_stride=wl.grid_stride, n_generate=n_generate)

    prompts = torch.from_numpy(make_prompt(wl, 5)).cuda()
    used = ctx()
    generate(used, prompts[:3].contiguous(), sample(11))
    again, counts_a, _ = generate(used, prompts[3:].contiguous(), sample(12))
    fresh, counts_f, _ = generate(ctx(), prompts[3:].contiguous(), sample(12))
    assert torch.equal(counts_a, counts_f)
    n = int(counts_f[0])
    assert torch.equal(again[:, :n], fresh[:, :n])


def test_tiny_fp32_full_generation():
    """The tiny fp32 configuration end to end: 256 tokens, W = 16, top-k 64, random initialisation."""
    wl = WORKLOADS["tiny"]
    ctx, seqs, steps, out = run_lockstep(wl)
    s = seqs[0]
    assert s.st.n == wl.prompt_len + wl.n_generate
    assert steps <= wl.n_generate
    assert s.max_logit_err <= 1e-4
    assert s.stats.flagged <= max(3, 0.02 * s.stats.decisions), s.stats
    # a finished sequence: further steps fix nothing and say so
    ctx.step(out)
    h = out.host()
    assert h["n_committed"][0] == 0 and h["flags"][0] & B.SJD_FLAG_DONE
    assert h["total_committed"][0] == wl.prompt_len + wl.n_generate


@pytest.mark.parametrize("init", [INIT_COPY_ABOVE, INIT_COPY_LEFT, INIT_RESAMPLE_LEFT, INIT_RESAMPLE_ABOVE])
def test_tiny_spatial_initialisation(init):
    wl = WORKLOADS["tiny"]
    run_lockstep(wl, init=init, n_generate=100)


def test_small_bf16_initialisation_from_the_prediction_above():
    """Sec. 4.2 (d) on the bf16 model with a grid row shorter than the window (stride 5, W = 16): the row
    above is sometimes a row of the pass just verified and sometimes a retained row of the ring, and a
    retained row serves as the draft's law on the register-resident verification route."""
    wl = WORKLOADS["small-bf16"].with_(grid_stride=5)
    ctx, seqs, steps, out = run_lockstep(wl, batch=2, init=INIT_RESAMPLE_ABOVE, n_generate=60)
    assert steps <= 60
    wl = WORKLOADS["small-bf16"]    # stride 16 = W: every source row comes from the ring
    ctx, seqs, steps, out = run_lockstep(wl, init=INIT_RESAMPLE_ABOVE, n_generate=60, schedule=2)
    assert steps <= 60


def test_resample_above_needs_a_ring():
    wl = WORKLOADS["tiny"]
    ctx = B.Context(B.make_model_cfg(wl, 1, 64, 8, max_ring=10), B.weights_to_device(make_weights(wl)))
    with pytest.raises(B.SJDError) as e:
        ctx.prefill(torch.from_numpy(make_prompt(wl, 1)).cuda(),
                    B.make_sample_cfg(top_k=10, window=8, n_generate=20, init=B.SJD_INIT_RESAMPLE_ABOVE, grid_stride=16))
    assert e.value.status == B.SJD_ERR_CAPACITY


@pytest.mark.parametrize("schedule", [0, 2])
def test_small_bf16_initialisation_from_the_left_neighbours_prediction(schedule):
    """Sec. 4.2 (c) on the bf16 model (rows verified on the register-resident route, new slots drawn from
    them by the sequence's last block), with and without refinement: without it every slot after the
    rejection is new and draws from the row that predicted its own left neighbour."""
    wl = WORKLOADS["small-bf16"]
    ctx, seqs, steps, out = run_lockstep(wl, batch=2, init=INIT_RESAMPLE_LEFT, n_generate=60, schedule=schedule)
    kinds = out.host()["q_kind"]
    assert steps <= 60


def test_tiny_batch_of_three_and_ragged_window():
    """Independent sequences in one batch; window 11 does not divide anything; sequence ids offset."""
    wl = WORKLOADS["tiny"]
    ctx, seqs, steps, _ = run_lockstep(wl, batch=3, window=11, n_generate=61, seq_base=5)
    assert all(s.st.n == wl.prompt_len + 61 for s in seqs)


@pytest.mark.parametrize("name,over,lens,kv_pages", [
    ("tiny", {}, (16, 5, 11), 0), ("small-bf16", {}, (24, 7, 1), 0),
    ("tiny", {}, (70, 5, 130), 6), ("small-bf16", {}, (100, 7, 64), 6),
    ("small-bf16", dict(head_dim=128, n_heads=4, n_kv_heads=2), (90, 130), 6)])
def test_ragged_prompts(name, over, lens, kv_pages):
    """Prompts of different lengths in one batch (sjd_prefill_ragged): every sequence keeps its own positions
    and finishes on its own; lock-step with one checker per sequence, each on its own prompt.  With kv_pages the
    cache is paged: the sequences' rows sit in pool pages handed out at pre-fill (a sequence's pages are not
    where a contiguous layout would put them, and its rows cross page boundaries), which the oracle knows
    nothing about, so agreement shows the paging changes no result."""
    wl = WORKLOADS[name].with_(**over)
    n_generate, window = 40, wl.window
    weights = make_weights(wl, gain_jitter=0.1)
    batch, stride = len(lens), max(lens)
    prompt = make_prompt(wl.with_(prompt_len=stride), batch)
    cfg = B.make_model_cfg(wl, max_batch=batch, max_seq=stride + n_generate + 8, max_window=window,
                           kv_pages=kv_pages)
    ctx = B.Context(cfg, B.weights_to_device(weights))
    sample = B.make_sample_cfg(temperature=wl.temperature, top_k=wl.top_k, seed=wl.philox_seed, window=window,
                               init=INIT_COPY_ABOVE, grid_stride=wl.grid_stride, n_generate=n_generate)
    if kv_pages:   # one page short: refused before anything is enqueued
        small = B.Context(B.make_model_cfg(wl, max_batch=batch, max_seq=stride + n_generate + 8, max_window=window,
                                           kv_pages=kv_pages - 1), B.weights_to_device(weights))
        with pytest.raises(B.SJDError) as e:
            small.prefill_ragged(torch.from_numpy(prompt).cuda(), lens, sample)
        assert e.value.status == B.SJD_ERR_CAPACITY
        del small
    scfg = SampleCfg(temperature=wl.temperature, top_k=wl.top_k, seed=wl.philox_seed, window=window,
                     init=INIT_COPY_ABOVE, grid_stride=wl.grid_stride, n_generate=n_generate, logits_dtype=wl.dtype)
    ctx.prefill_ragged(torch.from_numpy(prompt).cuda(), lens, sample)
    out = B.StepOut(batch, window)
    ctx.get_window(out)
    h = out.host()
    seqs = [LockStepSequence(wl.with_(prompt_len=lens[b]), weights, prompt[b][:lens[b]], scfg, b, LOGIT_TOL[wl.dtype])
            for b in range(batch)]
    for b, s in enumerate(seqs):
        s.check_window(h["draft"][b], h["q_kind"][b], h["q_draft"][b], h["total_committed"][b])
    steps = 0
    while any(s.st.n < lens[b] + n_generate for b, s in enumerate(seqs)):
        ctx.step(out)
        logits = ctx.peek_logits().to(torch.float64).cpu().numpy()
        h = out.host()
        for b, s in enumerate(seqs):
            s.step(logits[b], {k: v[b] for k, v in h.items()})
        steps += 1
        assert steps <= n_generate
    assert ctx.device_status() == B.SJD_OK
    assert [s.st.n for s in seqs] == [l + n_generate for l in lens]


def test_tiny_window_of_one_is_ordinary_sampling():
    wl = WORKLOADS["tiny"]
    ctx, seqs, steps, _ = run_lockstep(wl, window=1, n_generate=24)
    assert steps == 24


def test_tiny_top1_is_greedy_decoding():
    from oracle.model import OracleModel
    from oracle.sjd import CachedModel, greedy_ar_generate
    from tests.parity_util import oracle_model_cfg
    wl = WORKLOADS["tiny"]
    ctx, seqs, steps, _ = run_lockstep(wl, n_generate=48, top_k=1, gain_jitter=0.0)
    weights = make_weights(wl)
    greedy = greedy_ar_generate(list(make_prompt(wl)[0]),
                                CachedModel(OracleModel(oracle_model_cfg(wl), weights), 80), 48)
    assert seqs[0].st.committed[wl.prompt_len:] == greedy
    assert steps <= 48


def run_lockstep_guided(wl, images, guidance, max_steps=None, init=INIT_RANDOM, window=None, n_generate=None, schedule=0,
                        kv_pages=0):
    """Lock-step under classifier-free guidance: 2 * images sequences in the library (conditional and
    unconditional stream of each image, prompts of one length with different tokens), one checker per image."""
    window = window or wl.window
    n_generate = wl.n_generate if n_generate is None else n_generate
    weights = make_weights(wl, gain_jitter=0.1)
    prompt = make_prompt(wl, 2 * images)       # rows 2i / 2i+1: conditional / unconditional prompt of image i
    cfg = B.make_model_cfg(wl, max_batch=2 * images, max_seq=wl.prompt_len + n_generate + 8, max_window=window,
                           max_ring=wl.grid_stride + window if init == INIT_RESAMPLE_ABOVE else 0, kv_pages=kv_pages)
    ctx = B.Context(cfg, B.weights_to_device(weights))
    sample = B.make_sample_cfg(temperature=wl.temperature, top_k=wl.top_k, seed=wl.philox_seed, window=window,
                               init=init, grid_stride=wl.grid_stride, n_generate=n_generate, guidance=guidance,
                               schedule=schedule)
    scfg = SampleCfg(temperature=wl.temperature, top_k=wl.top_k, seed=wl.philox_seed, window=window, init=init,
                     grid_stride=wl.grid_stride, n_generate=n_generate, logits_dtype=wl.dtype, schedule=schedule)
    ctx.prefill(torch.from_numpy(prompt).cuda(), sample)
    out = B.StepOut(images, window)
    ctx.get_window(out)
    h = out.host()
    seqs = [LockStepSequence(wl, weights, prompt[2 * i], scfg, i, LOGIT_TOL[wl.dtype], guidance=guidance,
                             prompt_uncond=prompt[2 * i + 1]) for i in range(images)]
    for i, s in enumerate(seqs):
        s.check_window(h["draft"][i], h["q_kind"][i], h["q_draft"][i], h["total_committed"][i])
    steps, total = 0, wl.prompt_len + n_generate
    while any(s.st.n < total for s in seqs):
        ctx.step(out)
        logits = ctx.peek_logits().to(torch.float64).cpu().numpy()
        h = out.host()
        for i, s in enumerate(seqs):
            s.step((logits[2 * i], logits[2 * i + 1]), {k: v[i] for k, v in h.items()})
        steps += 1
        assert steps <= n_generate
        if max_steps and steps >= max_steps:
            break
    assert ctx.device_status() == B.SJD_OK
    return seqs, steps


def test_tiny_guided_generation():
    """Classifier-free guidance (weight 3.0) on the tiny fp32 model: two streams per image, one shared
    verification on the mixed rows; two images, 60 tokens each, copied-token initialisation."""
    wl = WORKLOADS["tiny"]
    seqs, steps = run_lockstep_guided(wl, images=2, guidance=3.0, n_generate=60, init=INIT_COPY_LEFT)
    for s in seqs:
        assert s.st.n == wl.prompt_len + 60
        assert s.stats.flagged <= max(3, 0.03 * s.stats.decisions), s.stats


@pytest.mark.parametrize("name,init,schedule,kv_pages", [
    ("tiny", INIT_RESAMPLE_ABOVE, 0, 0), ("small-bf16", INIT_RESAMPLE_ABOVE, 0, 0),
    ("small-bf16", INIT_RESAMPLE_LEFT, 2, 0), ("tiny", INIT_RANDOM, 1, 0),
    ("small-bf16", INIT_RESAMPLE_ABOVE, 0, 8), ("tiny", INIT_COPY_ABOVE, 0, 8)])
def test_guided_generation_with_the_other_options(name, init, schedule, kv_pages):
    """Guidance together with the initialisations that draw from predicted distributions (the ring then
    holds mixed rows, one per image position), with the no-refinement ablation, with the Jacobi schedule and
    with the paged cache (four streams of two pages each)."""
    wl = WORKLOADS[name]
    seqs, steps = run_lockstep_guided(wl, images=2, guidance=3.0, n_generate=50, init=init, schedule=schedule,
                                      kv_pages=kv_pages)
    for s in seqs:
        assert s.st.n == wl.prompt_len + 50


def test_small_bf16_guided_generation():
    """The same on the small bf16 model (tensor-core pipeline, register-resident verification route):
    the mixed row is rounded to bf16 before the top-k threshold is taken."""
    wl = WORKLOADS["small-bf16"]
    seqs, steps = run_lockstep_guided(wl, images=2, guidance=3.0, n_generate=80)
    for s in seqs:
        assert s.max_logit_err <= 2e-2
        assert s.stats.flagged <= max(3, 0.03 * s.stats.decisions), s.stats


@pytest.mark.parametrize("name,batch", [("tiny", 1), ("small-bf16", 2)])
def test_jacobi_schedule(name, batch):
    """Sec. 3.2 on the same kernels: every slot re-drawn each pass with the uniform of its position, the
    unchanged prefix fixed.  Lock-step with the checker; on the fp32 model the finished image must also
    be the one ordinary sampling draws from the same uniforms."""
    from oracle.model import OracleModel
    from oracle.sjd import SCHEDULE_JACOBI, CachedModel, ar_generate
    from tests.parity_util import oracle_model_cfg
    wl = WORKLOADS[name]
    n_gen = 48
    ctx, seqs, steps, _ = run_lockstep(wl, batch=batch, n_generate=n_gen, schedule=SCHEDULE_JACOBI, gain_jitter=0.0)
    assert steps <= n_gen
    if wl.dtype == "f32" and seqs[0].stats.flagged == 0:
        scfg = SampleCfg(temperature=wl.temperature, top_k=wl.top_k, seed=wl.philox_seed, n_generate=n_gen,
                         logits_dtype=wl.dtype)
        model = CachedModel(OracleModel(oracle_model_cfg(wl), make_weights(wl)), wl.prompt_len + n_gen + 1)
        plain, _ = ar_generate(list(make_prompt(wl)[0]), model, scfg, wl.vocab, fixed_step=0)
        assert seqs[0].st.committed[wl.prompt_len:] == plain


@pytest.mark.parametrize("name,init", [("tiny", INIT_RANDOM), ("small-bf16", INIT_COPY_LEFT)])
def test_no_refinement_schedule(name, init):
    """The ablation without Eq. 3: after the first rejection every remaining slot is initialised afresh."""
    from oracle.sjd import SCHEDULE_NO_REFINE
    wl = WORKLOADS[name]
    ctx, seqs, steps, out = run_lockstep(wl, n_generate=40, schedule=SCHEDULE_NO_REFINE, init=init)
    assert steps <= 40
    assert not np.any(out.host()["q_kind"] == B.SJD_Q_ROW)


@pytest.mark.parametrize("name,n_generate", [("tiny", 60), ("small-bf16", 80), ("7b-2l", 0)])
def test_qk_norm_variant(name, n_generate):
    """The QK-norm variant of the decoder (per-head RMS normalisation of q and k before the rotary step, the
    Chameleon family): generic kernels (tiny fp32), tensor-core pipeline with head_dim 64 (small bf16) and
    with head_dim 128 (7B layer shapes, two layers, three steps)."""
    wl = WORKLOADS[name]
    if n_generate:
        ctx, seqs, steps, _ = run_lockstep(wl, batch=2 if name != "tiny" else 1, n_generate=n_generate, qk_norm=True)
    else:
        ctx, seqs, steps, _ = run_lockstep(wl, max_steps=3, gain_jitter=0.0, qk_norm=True)
    for s in seqs:
        assert s.max_logit_excess <= LOGIT_TOL[wl.dtype]


def test_small_bf16_gqa_generation():
    """bf16 storage, grouped-query attention, sizes that are not multiples of the tile sizes."""
    wl = WORKLOADS["small-bf16"]
    ctx, seqs, steps, _ = run_lockstep(wl, batch=2)
    for s in seqs:
        assert s.max_logit_err <= 2e-2
        assert s.stats.flagged <= max(3, 0.03 * s.stats.decisions), s.stats


@pytest.mark.parametrize("guidance,init", [(0.0, INIT_RESAMPLE_ABOVE), (3.0, INIT_RESAMPLE_LEFT), (3.0, INIT_RANDOM)])
def test_small_bf16_vocabulary_longer_than_the_registers(guidance, init):
    """A 70016-entry vocabulary on the small bf16 model: every logits row is verified on the streamed form of
    the register route (two segments), with cached statistics of the previous rows, with the rows of the two
    guidance streams mixed as they are loaded, and with retained rows as the drafts' laws."""
    wl = WORKLOADS["small-bf16"].with_(vocab=70016, top_k=2000)
    if guidance:
        seqs, steps = run_lockstep_guided(wl, images=1, guidance=guidance, n_generate=40, init=init)
    else:
        _, seqs, steps, _ = run_lockstep(wl, batch=2, init=init, n_generate=40)
    for s in seqs:
        assert s.st.n == wl.prompt_len + 40
        assert s.max_logit_err <= 2e-2
        assert s.stats.flagged <= max(3, 0.04 * s.stats.decisions), s.stats


def test_small_bf16_128_rows():
    """8 images x W = 16 = 128 rows per pass: the largest single slab (256 MMA columns, two-stage ring) through
    pre-fill and three steps."""
    wl = WORKLOADS["small-bf16"]
    ctx, seqs, steps, _ = run_lockstep(wl, batch=8, max_steps=3)
    for s in seqs:
        assert s.max_logit_err <= 2e-2
        assert s.stats.flagged <= max(3, 0.03 * s.stats.decisions), s.stats


def test_small_bf16_many_rows():
    """20 images x W = 16 = 320 rows per pass: the token-slab form of the projections (three slabs of
    112 rows) through pre-fill and three steps."""
    wl = WORKLOADS["small-bf16"]
    ctx, seqs, steps, _ = run_lockstep(wl, batch=20, max_steps=3)
    for s in seqs:
        assert s.max_logit_err <= 2e-2
        assert s.stats.flagged <= max(3, 0.03 * s.stats.decisions), s.stats


@pytest.mark.parametrize("name,batch,prompt_len", [
    ("small-bf16", 1, 1300),   # 21 segments of 64 positions: two passes of the tensor-core pipeline
    ("small-bf16", 3, 66),     # 65 rows each: segments of 32 or 16, several per sequence in one pass
    ("small-bf16", 2, 2),      # a single row per sequence
    ("tiny", 2, 200),          # generic pipeline: two passes of at most 256 rows
])
def test_prefill_passes(name, batch, prompt_len):
    """Pre-fill packs segments of the prompts into passes: segment and pass boundaries, one-row prompts."""
    run_lockstep(WORKLOADS[name].with_(prompt_len=prompt_len), batch=batch, n_generate=40, max_steps=2)


def report_depth(label, seq):
    """One line per cache reading of the checker, for the depth table of the design notes."""
    print()
    print(seq.errors.line("%s, checker cache rounded to bf16" % label))
    if seq.errors_plain is not None:
        print(seq.errors_plain.line("%s, checker cache unrounded (plain definition)" % label))


@pytest.mark.parametrize("name,layers,steps", [("7b", 2, 4), ("8b-gqa", 2, 3), ("7b", 8, 2)])
def test_large_shapes_reduced_depth(name, layers, steps):
    """The 7B / 8B-GQA layer shapes (d 4096, SwiGLU 11008 / 14336, vocab 65536 / 184320, W 32 / 64,
    top-k 2000 / 2048) at two and eight layers, a few lock-step steps: every logit within 2e-2 (plus
    half a unit in the last place of the stored bf16 value) of the checker whose cache is rounded to
    bf16; the error against the checker with an unrounded cache is printed beside it."""
    wl = WORKLOADS[name].with_(n_layers=layers)
    ctx, seqs, n, _ = run_lockstep(wl, max_steps=steps, gain_jitter=0.0, also_plain_cache=True)
    report_depth("%s at %d layers" % (name, layers), seqs[0])
    assert seqs[0].max_logit_excess <= 2e-2


@pytest.mark.parametrize("batch,window,prompt_len,init,steps", [
    (4, 8, 64, INIT_COPY_ABOVE, 3),    # small window, spatial initialisation (grid stride 49), 32 rows per pass
    (2, 64, 64, INIT_RANDOM, 2),       # widest window: 128 rows per pass, attention in 128 columns with a ring of three tiles
    (8, 32, 64, INIT_RANDOM, 2),       # 256 rows per pass: two token slabs per weight tile at the 7B widths
    (3, 24, 64, INIT_RANDOM, 2),       # 72 rows: a slab that is not a multiple of 16, shared units among its tiles
    (1, 32, 700, INIT_COPY_ABOVE, 2),  # long prefix: several key tiles per split-KV range, pre-fill in 22 chunks
])
def test_sweep_points_two_layers(batch, window, prompt_len, init, steps):
    """Points of the batch / window / prefix / initialisation sweep on the 7B layer shapes (two layers so
    that the checker stays affordable), in lock-step with the checker."""
    wl = WORKLOADS["7b-2l"].with_(prompt_len=prompt_len)
    ctx, seqs, n, _ = run_lockstep(wl, batch=batch, window=window, init=init, max_steps=steps, gain_jitter=0.0)
    assert n == steps
    for s in seqs:
        assert s.max_logit_excess <= 2e-2


@pytest.mark.parametrize("name,over,batch,window", [
    ("tiny", dict(n_heads=3, n_kv_heads=3, head_dim=62, d_model=250, vocab=1021), 1, 5),   # rows off 16 bytes, widths off the tiles
    ("tiny", {}, 5, 31),                                                                    # 155 rows: 16 x 32 and 32 x 32 tiles
    ("tiny", dict(ffn_hidden=1503, vocab=2050), 9, 31),                                     # 279 rows, the last tiles partly outside
    ("small-bf16", dict(ffn_hidden=1003, d_model=500, vocab=1501), 6, 33),                  # bf16, 198 rows, groups and single entries
    ("small-bf16", dict(ffn_hidden=1003, vocab=1001), 2, 7),                                # bf16, some matrices unaligned
])
def test_generic_projections(name, over, batch, window):
    """The generic pipeline (fused normalisation, residual and SwiGLU) on row counts and widths off its tiles."""
    ctx, seqs, n, _ = run_lockstep(WORKLOADS[name].with_(**over), batch=batch, window=window, n_generate=30, max_steps=3)
    assert ctx.info()["tensor_core_projections"] == 0


@pytest.mark.parametrize("over,qk_norm", [
    (dict(head_dim=96, n_heads=4, n_kv_heads=4, d_model=512), True),    # halves of 48 entries: two per lane, some idle
    (dict(head_dim=32, n_heads=16, n_kv_heads=4), False),              # halves of 16
])
def test_rotary_step_of_other_head_sizes(over, qk_norm):
    """The cache append of the tensor-core pipeline at head sizes without tensor-core attention."""
    ctx, seqs, n, _ = run_lockstep(WORKLOADS["small-bf16"].with_(**over), batch=2, n_generate=40, max_steps=2, qk_norm=qk_norm)
    assert ctx.info()["tensor_core_projections"] == 1 and ctx.info()["tensor_core_attention"] == 0


@pytest.mark.parametrize("name,batch,window,prompt_len", [
    ("7b-2l", 3, 5, 90),        # 15 rows
    ("7b-2l", 1, 9, 530),       # one sequence whose keys are spread over several CTAs and merged
    ("8b-gqa-2l", 2, 31, 70),   # 62 rows, four query heads per K/V head
])
def test_wide_layers_ragged_rows(name, batch, window, prompt_len):
    """Row counts off the 16-row grid on the 7B / 8B layer shapes."""
    ctx, seqs, n, _ = run_lockstep(WORKLOADS[name].with_(prompt_len=prompt_len), batch=batch, window=window, max_steps=2,
                                   gain_jitter=0.1)
    for s in seqs:
        assert s.max_logit_excess <= 2e-2


@pytest.mark.parametrize("name,steps", [("7b", 2), ("8b-gqa", 1)])
def test_full_depth(name, steps):
    """The full configurations (7B: 32 layers, vocab 65536, W = 32, the step the benchmark times; 8B with
    grouped-query heads: 32 layers, vocab 184320, W = 64) for the pre-fill and one or two lock-step
    iterations: every decision re-taken by the fp64 checker (exact), every logit of the windows compared
    with the checker under both readings of the cache (rounded to bf16 like the library's; unrounded).
    The rule at this depth, fixed: against the rounded-cache checker, 2e-2 (plus half a unit in the last
    place of the stored value) on all but one in a million logits, and 3e-2 on every one.  The error
    grows with the square root of the depth (two, eight and 32 layers are printed by this file) and the
    worst of 4 to 12 million logits sits at the 2e-2 bar at 32 layers.
    Needs ~40 GB of host memory for the checker's weights and cache."""
    import psutil
    if psutil.virtual_memory().available < 64 * 2 ** 30:
        pytest.skip("not enough host memory for the full-depth checker")
    wl = WORKLOADS[name]

    def every_logit_bar(self, diff, half_ulp):
        return diff > 3e-2 + half_ulp

    old = LockStepSequence.logit_failures
    LockStepSequence.logit_failures = every_logit_bar
    try:
        ctx, seqs, n, _ = run_lockstep(wl, max_steps=steps, gain_jitter=0.0, also_plain_cache=True)
    finally:
        LockStepSequence.logit_failures = old
    assert n == steps and seqs[0].steps == steps
    report_depth("%s at 32 layers" % name, seqs[0])
    e = seqs[0].errors
    assert e.beyond[2] <= e.total // 1000000, (e.beyond, e.total)


def test_api_errors_and_state():
    wl = WORKLOADS["tiny"]
    weights = B.weights_to_device(make_weights(wl))
    cfg = B.make_model_cfg(wl, max_batch=2, max_seq=64, max_window=8)
    ctx = B.Context(cfg, weights)
    with pytest.raises(B.SJDError) as e:
        ctx.step(None)
    assert e.value.status == B.SJD_ERR_STATE
    prompt = torch.from_numpy(make_prompt(wl, 2)).cuda()
    for kw, status in [(dict(window=9), B.SJD_ERR_CAPACITY), (dict(n_generate=60), B.SJD_ERR_CAPACITY),
                       (dict(temperature=0.0), B.SJD_ERR_BAD_ARG), (dict(top_k=0), B.SJD_ERR_BAD_ARG),
                       (dict(init=1, grid_stride=0), B.SJD_ERR_BAD_ARG)]:
        args = dict(top_k=10, window=8, n_generate=20)
        args.update(kw)
        with pytest.raises(B.SJDError) as e:
            ctx.prefill(prompt, B.make_sample_cfg(**args))
        assert e.value.status == status, kw
    bad = B.make_model_cfg(wl, max_batch=0, max_seq=64, max_window=8)
    assert B.sjd_workspace_bytes(bad) == 0
    with pytest.raises(B.SJDError):
        B.Context(B.make_model_cfg(wl.with_(head_dim=63), 1, 64, 8), weights)
    torch.cuda.synchronize()


@pytest.mark.parametrize("name,over", [("tiny", {}), ("small-bf16", {}), ("small-bf16", dict(ffn_hidden=1400))])
def test_bad_prompt_token_raises_the_flag(name, over):
    """A prompt token whose embedding is not a number makes every key it leaves in the cache one: the iterations of its sequence
    say so, those of the other sequence do not.  (Both pipelines, several key ranges: the long prompt's keys are in all of them.)"""
    wl = WORKLOADS[name].with_(**over)
    weights = make_weights(wl)
    weights["tok_emb"][7] = float("nan")
    prompt = torch.randint(8, wl.vocab, (2, 300), generator=torch.Generator().manual_seed(3), dtype=torch.int32)
    prompt[0, 40] = 7
    ctx = B.Context(B.make_model_cfg(wl, max_batch=2, max_seq=400, max_window=wl.window), B.weights_to_device(weights))
    ctx.prefill(prompt.cuda(), B.make_sample_cfg(top_k=50, window=wl.window, n_generate=40, seed=1))
    out = B.StepOut(2, wl.window)
    ctx.get_window(out)
    assert not (out.host()["draft"] == 7).any()   # (no draft of this seed is the bad token)
    ctx.step(out)
    flags = out.host()["flags"]
    assert flags[0] & B.SJD_FLAG_NONFINITE and not flags[1] & B.SJD_FLAG_NONFINITE
    logits = ctx.peek_logits()
    assert logits[0].isnan().all() and not logits[1].isnan().any()
    assert ctx.device_status() == B.SJD_OK


@pytest.mark.parametrize("refused", [
    dict(batch=1, seed=5, n_generate=250),   # five pages needed, four there
    dict(batch=2, seed=2, n_generate=120),   # six pages for a larger batch
])
def test_refused_prefill_leaves_the_generation_alone(refused):
    """A pre-fill that the paged cache cannot hold is refused before anything of the context changes: the generation
    under way goes on to the tokens that it yields undisturbed."""
    wl = WORKLOADS["small-bf16"]
    weights = B.weights_to_device(make_weights(wl))
    prompt = torch.from_numpy(make_prompt(wl, 2)).cuda()
    tokens = []
    for disturbed in (False, True):
        ctx = B.Context(B.make_model_cfg(wl, 2, 320, wl.window, 0, 4), weights)
        ctx.prefill(prompt[:1].contiguous(), B.make_sample_cfg(top_k=wl.top_k, seed=2, window=wl.window, n_generate=100))
        out = B.StepOut(1, wl.window)
        for step in range(40):
            if disturbed and step in (1, 7):
                with pytest.raises(B.SJDError) as e:
                    ctx.prefill(prompt[:refused["batch"]].contiguous(),
                                B.make_sample_cfg(top_k=wl.top_k, seed=refused["seed"], window=wl.window,
                                                  n_generate=refused["n_generate"]))
                assert e.value.status == B.SJD_ERR_CAPACITY
            ctx.step(out)
        tokens.append([t.cpu() for t in (*ctx.get_tokens(), ctx.peek_logits())])
    for a, b in zip(*tokens):
        assert torch.equal(a, b)


def test_contexts_on_two_streams():
    """Two contexts of 80 rows per pass (projections on CTA pairs that share the units of a partial last round) step at the
    same time on two streams: each yields what it yields alone."""
    wl = WORKLOADS["small-bf16"]
    weights = B.weights_to_device(make_weights(wl))
    prompt = torch.from_numpy(make_prompt(wl, 5)).cuda()

    def run(seed, got):
        ctx = B.Context(B.make_model_cfg(wl, 5, 320, wl.window), weights)
        ctx.prefill(prompt, B.make_sample_cfg(top_k=wl.top_k, seed=seed, window=wl.window, n_generate=250))
        for _ in range(150):
            ctx.step()
        got[seed] = [t.cpu() for t in (*ctx.get_tokens(), ctx.peek_logits())]
        assert ctx.device_status() == B.SJD_OK

    alone, together = {}, {}
    for seed in (1, 2):
        run(seed, alone)
    run_in_threads(*[lambda seed=seed: run(seed, together) for seed in (1, 2)])
    for seed in (1, 2):
        for a, b in zip(alone[seed], together[seed]):
            assert torch.equal(a, b)
