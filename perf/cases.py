"""Cases that the performance of this framework is measured on: what its users have it do, through the public calls.

A case is one pass of such a use: whole sentences decoded (`AggressiveDecoder.generate` / `generate_device`), a loop that the
user's own program drives block by block (`encode`, `draft_block`, `verify_block`, `commit`), or one of the operator-level
calls (`linear`, `vocab_argmax`, `vocab_argmax_static`).  Model shapes, batch sizes, source lengths and block sizes are
those of the workload recipes and shapes in `paper_2205_10350_b200/synth.py`, and odd sizes between them.

Models.  Plain random weights make a model that repeats its last token whatever the source says.  A trained corrector or
translator instead follows its source and departs from it here and there, with clear gaps between the best and the second
best score; the method lives on that.  `_weights` therefore adds to the random tensors what makes a model do so: an
undisturbed positional subspace, a last cross-attention that looks up the source position being decoded and carries its
token over, and embeddings in which every sixteenth id is a weaker variant of its successor, so that a source holding the
variant is rewritten.  The drafter is such a model too, non-autoregressive and with twice as many variants, so that it
agrees with the verifier on about 85 % of the tokens.  Decoding then runs as in earnest: long accepted blocks, bifurcations
at the rewritten tokens, suffix matches in the source, [EOS] at the end.

A user's program keeps one decoder per model and capacity and sends it sentence after sentence; so do these cases.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2205_10350_b200 import binding, synth

DEV = "cuda:0"
MODELS = {"tiny": synth.TINY, "base": synth.BASE, "big": synth.BIG, "deep_enc": synth.DEEP_ENC, "bart_sized": synth.BART_BASE_SIZED}
BETA, TAU = 3, 4.0            # relaxed verification: the draft among the three best and at most 4.0 below the best score
EDIT_RATE = 0.09              # share of source tokens that the verifier rewrites
DRAFT_AGREEMENT = 0.85        # share of tokens that the drafter chooses like the verifier
STEP_ROUNDS = 3               # rounds of a block-by-block loop


def listed():
    return [
        # recipe 1: the smallest model, FP32 arithmetic, one short sentence: launches and latency, nothing else
        dict(name="tiny_fp32_iad_b1", kind="generate", model="tiny", mode="IAD", batch=1, src_lo=16, src_hi=16, max_out=24, k=17, api="host"),
        # recipe 2: grammatical error correction of single sentences as they come in, host arrays in and out
        dict(name="base_iad_b1", kind="generate", model="base", mode="IAD", batch=1, src_lo=12, src_hi=40, max_out=0, k=64, api="host"),
        # recipe 3: the same model over a ragged batch of 32 sentences, arrays resident on the device
        dict(name="base_iad_b32", kind="generate", model="base", mode="IAD", batch=32, src_lo=10, src_hi=64, max_out=0, k=64, api="device"),
        # recipe 4: translation of single sentences with the big model and its drafter
        dict(name="big_gad_b1", kind="generate", model="big", mode="GAD", batch=1, src_lo=20, src_hi=50, max_out=0, k=25, api="host"),
        # recipe 5: summarisation, long sources in small batches, drafter
        dict(name="base_gad_b8_s400", kind="generate", model="base", mode="GAD", batch=8, src_lo=400, src_hi=400, max_out=80, k=25, api="device"),
        # plain greedy decoding (block size 1): what the method is compared with, and what a user without drafts runs
        dict(name="big_greedy_b4", kind="generate", model="big", mode="IAD", batch=4, src_lo=20, src_hi=50, max_out=0, k=1, api="device"),
        # relaxed verification of drafts that the user's program brings along, a model of another width, odd sizes
        dict(name="bart_gadpp_b3_s150", kind="generate", model="bart_sized", mode="GAD++", batch=3, src_lo=90, src_hi=150, max_out=61, k=30, api="host"),
        # the user's own loop over the block-level calls, deep encoder and shallow decoder, odd batch
        dict(name="deep_enc_steps_b5", kind="steps", model="deep_enc", drafter=False, batch=5, src_lo=25, src_hi=75, k=33),
        # output projection with arg-max over the rows of an ordinary batch
        dict(name="argmax_bf16_m600", kind="argmax", dtype="bf16", rows=600, d=512, vocab=32000, static=False),
        # the same for a caller that may not allocate, a handful of rows, ragged vocabulary
        dict(name="argmax_static_bf16_m7", kind="argmax", dtype="bf16", rows=7, d=768, vocab=50265, static=True),
        # one projection of the feed-forward sublayer over a large batch, and an FP32 one over an odd number of rows
        dict(name="linear_bf16_m1800", kind="linear", dtype="bf16", rows=1800, k_in=2048, n_out=512),
        dict(name="linear_fp32_m333", kind="linear", dtype="fp32", rows=333, k_in=512, n_out=2048),
    ]


def _log_int(rng, lo, hi):
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_once(rng):
    kind = rng.choice(["generate"] * 6 + ["steps", "argmax", "linear"])
    if kind == "generate":
        model = rng.choice(["tiny", "base", "base", "big", "deep_enc", "bart_sized"])
        mode = rng.choice(["IAD", "IAD", "GAD", "GAD", "GAD++"])
        small = model == "tiny"
        batch = _log_int(rng, 1, 6 if small else 32)
        hi = _log_int(rng, 12, 40 if small else 400)
        lo = rng.randint(max(4, hi // 4), hi)
        # [EOS] ends the output of a short source; long sources are summarised
        max_out = 0 if hi <= 80 else rng.randint(20, 80)
        k = 1 if rng.random() < 0.15 else _log_int(rng, 4, 64)
        return dict(kind=kind, model=model, mode="IAD" if k == 1 else mode, batch=batch, src_lo=lo, src_hi=hi, max_out=max_out, k=k,
                    api=rng.choice(["host", "device"]))
    if kind == "steps":
        hi = _log_int(rng, 24, 300)
        return dict(kind=kind, model=rng.choice(["base", "deep_enc", "bart_sized"]), drafter=rng.random() < 0.5, batch=_log_int(rng, 1, 16),
                    src_lo=rng.randint(max(20, hi // 2), hi), src_hi=hi, k=_log_int(rng, 5, 50))
    if kind == "argmax":
        d, vocab = rng.choice([(512, 32000), (1024, 32000), (768, 50265)])
        static = rng.random() < 0.4
        fp32 = rng.random() < 0.25
        return dict(kind=kind, dtype="fp32" if fp32 else "bf16", rows=_log_int(rng, 1, 250 if static else (100 if fp32 else 3000)), d=d,
                    vocab=32000 if static and vocab > 32000 else vocab, static=static)
    fp32 = rng.random() < 0.4
    k_in, n_out = rng.choice([(512, 1536), (512, 2048), (2048, 512), (1024, 4096), (4096, 1024), (768, 3072), (1024, 1000)])
    return dict(kind=kind, dtype="fp32" if fp32 else "bf16", rows=_log_int(rng, 1, 700 if fp32 else 4000), k_in=k_in, n_out=n_out)


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


@functools.lru_cache(maxsize=None)
def _largest():
    return max(_cost(c) for c in listed())


def draw(rng):
    while True:
        case = _draw_once(rng)
        if _cost(case) <= _largest():
            return case


# ------------------------------------------------------------------------------------------------------
# models and handles, built once and kept
# ------------------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=3)
def _weights(model, drafter):
    """Host weights of a model that follows its source (see the top of this file)."""
    shape = MODELS[model]
    d, heads, vocab = shape.d_model, shape.n_heads, shape.vocab
    dh = d // heads
    gen = torch.Generator(DEV).manual_seed(2 * sorted(MODELS).index(model) + int(drafter))
    w = {}
    for name, dims in synth.weight_names(shape):
        t = torch.randn(dims, generator=gen, device=DEV) * (d ** -0.5 if name == "emb" else 0.02)
        if name.endswith(".g"):
            t += 1.0
        if name.endswith(".o.W") or name.endswith(".ffn2.W"):
            t *= 0.5
            t[:, :dh] = 0.0                    # the first head's dimensions carry the position alone
        w[name] = t
    w["emb"][:, :dh] = 0.0
    ids = torch.arange(synth.FIRST_ORDINARY_ID, vocab - 1, device=DEV)
    variant = ids[(ids % 8 == 0) if drafter else (ids % 16 == 0)]
    w["emb"][variant] = 0.8 * w["emb"][variant + 1]
    # last cross-attention: every head compares positions (the drafter reads one position back: its mask slot for output
    # token t sits at position t + 1) and carries its share of the source token over
    freq = torch.exp(-math.log(10000.0) * torch.arange(0, dh, 2) / d)
    q, k = torch.zeros(d, d), torch.zeros(d, d)
    for h in range(heads):
        for i in range(dh // 2):
            if freq[i] < 0.5:
                continue
            a, b = 2 * i, 2 * i + 1
            c, s = (math.cos(freq[i]), math.sin(freq[i])) if drafter else (1.0, 0.0)
            k[a, h * dh + a] = k[b, h * dh + b] = 6.0
            q[a, h * dh + a], q[b, h * dh + a] = 6.0 * c, -6.0 * s
            q[b, h * dh + b], q[a, h * dh + b] = 6.0 * c, 6.0 * s
    last = f"dec.{shape.n_dec - 1}.cross"
    w[f"{last}.q.W"], w[f"{last}.k.W"] = q.to(DEV), k.to(DEV)
    w[f"{last}.v.W"], w[f"{last}.o.W"] = torch.eye(d, device=DEV), 4.0 * torch.eye(d, device=DEV)
    if shape.dtype == "bf16":
        w = {n: t.bfloat16().float() for n, t in w.items()}
    return {n: t.cpu().numpy() for n, t in w.items()}


@functools.lru_cache(maxsize=None)
def _decoder(model, drafter, max_batch, max_src, max_tgt, kmax, relaxed):
    dec = binding.AggressiveDecoder(MODELS[model], _weights(model, False), _weights(model, True) if drafter else None,
                                    max_batch=max_batch, max_src=max_src, max_tgt=max_tgt, kmax=kmax, device=DEV)
    if relaxed:
        dec.set_acceptance(BETA, TAU)
    return dec


@functools.lru_cache(maxsize=None)
def _matrix(rows, cols, dtype):
    """A weight matrix of an operator-level call: one per shape, kept like a model's."""
    gen = torch.Generator(DEV).manual_seed(rows * 7919 + cols)
    return (torch.randn((rows, cols), generator=gen, device=DEV) * 0.02).to(dtype)


def _max_tgt(case):
    return case["max_out"] if case["max_out"] > 0 else case["src_hi"]


def _sources(case, rng):
    shape = MODELS[case["model"]]
    lens = rng.integers(case["src_lo"], case["src_hi"] + 1, size=case["batch"]).astype(np.int32)
    src = np.full((case["batch"], case["src_hi"]), synth.PAD, np.int32)
    for b, n in enumerate(lens):
        src[b, :n] = rng.integers(synth.FIRST_ORDINARY_ID, shape.vocab, size=int(n))
        src[b, n - 1] = synth.EOS
    return src, lens


# ------------------------------------------------------------------------------------------------------
# what a user has in hand, and one pass
# ------------------------------------------------------------------------------------------------------
def prepare(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "generate":
        cap, gad = _max_tgt(case), case["mode"] == "GAD"
        k = min(case["k"], cap)
        dec = _decoder(case["model"], gad, case["batch"], case["src_hi"], cap, k, case["mode"] == "GAD++")
        src, lens = _sources(case, rng)
        max_len = np.minimum(lens, cap).astype(np.int32) if case["max_out"] == 0 else np.full(case["batch"], cap, np.int32)
        stream = None
        if case["mode"] == "GAD++":           # the drafts that come along: the source itself, position by position
            stream = np.full((case["batch"], cap), synth.PAD, np.int32)
            stream[:, : min(cap, src.shape[1])] = src[:, :cap]
        state = dict(kind="generate", dec=dec, api=case["api"], cap=cap,
                     opts=dict(mode="IAD" if case["mode"] == "IAD" else "GAD", k=k, run_drafter=gad))
        if case["api"] == "host":
            state.update(src=src, lens=lens, max_len=max_len, stream=stream)
        else:
            t = lambda a: None if a is None else torch.tensor(a, device=DEV)
            state.update(src=t(src), lens=t(lens), max_len=t(max_len), stream=t(stream),
                         out=torch.zeros((case["batch"], cap), dtype=torch.int32, device=DEV),
                         out_len=torch.zeros(case["batch"], dtype=torch.int32, device=DEV))
        return state
    if case["kind"] == "steps":
        cap = min(case["src_hi"], 3 * case["k"])
        dec = _decoder(case["model"], case["drafter"], case["batch"], case["src_hi"], cap, min(case["k"], cap), False)
        src, lens = _sources(case, rng)
        return dict(kind="steps", dec=dec, drafter=case["drafter"], src=src, lens=lens)
    gen = torch.Generator(DEV).manual_seed(seed)
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    if case["kind"] == "argmax":
        x = torch.randn((case["rows"], case["d"]), generator=gen, device=DEV).to(dtype)
        return dict(kind="argmax", x=x, emb=_matrix(case["vocab"], case["d"], dtype), static=case["static"],
                    out=torch.zeros(case["rows"], dtype=torch.int32, device=DEV))
    x = torch.randn((case["rows"], case["k_in"]), generator=gen, device=DEV).to(dtype)
    bias = torch.randn(case["n_out"], generator=gen, device=DEV) * 0.02
    return dict(kind="linear", x=x, W=_matrix(case["n_out"], case["k_in"], dtype), bias=bias)


def run(state):
    if state["kind"] == "generate":
        dec, opts = state["dec"], state["opts"]
        if state["api"] == "host":
            out = np.zeros((len(state["lens"]), state["cap"]), np.int32)
            out_len = np.zeros(len(state["lens"]), np.int32)
            rows, _ = dec.generate(state["src"], state["lens"], max_len=state["max_len"], draft_override=state["stream"], out=out,
                                   out_len=out_len, **opts)
            tokens = np.full_like(out, synth.PAD)
            for b, r in enumerate(rows):
                tokens[b, : len(r)] = r
            return dict(tokens=tokens, length=out_len)
        dec.generate_device(state["src"], state["lens"], state["out"], state["out_len"], max_len_t=state["max_len"],
                            override_t=state["stream"], **opts)
        # entries past a row's length are not part of the result
        keep = torch.arange(state["cap"], device=DEV)[None, :] < state["out_len"][:, None]
        return dict(tokens=torch.where(keep, state["out"], synth.PAD), length=state["out_len"])
    if state["kind"] == "steps":
        dec, src, lens = state["dec"], state["src"], state["lens"]
        B, kmax = len(lens), dec.kmax
        dec.encode(src, lens)
        done, over = np.zeros(B, np.int32), np.zeros(B, bool)
        chosen, accepted = [], []
        for _ in range(STEP_ROUNDS):
            room = np.where(over, 0, np.minimum(lens, dec.max_tgt) - done)
            if state["drafter"]:
                drafts, k = dec.draft_block(kmax)
                k = np.minimum(k, room).astype(np.int32)
            else:                             # drafts copied from the source, position by position
                k = np.minimum(room, kmax).astype(np.int32)
                drafts = np.full((B, kmax), -1, np.int32)
                for b in range(B):
                    drafts[b, : k[b]] = src[b, done[b]: done[b] + k[b]]
            ids, n = dec.verify_block(drafts, k)
            dec.commit()
            done = done + n
            for b in range(B):
                over[b] |= k[b] == 0 or done[b] >= lens[b] or ids[b, max(int(n[b]) - 1, 0)] == synth.EOS
            chosen.append(np.where(np.arange(kmax)[None, :] < k[:, None], ids, synth.PAD))
            accepted.append(n)
        return dict(chosen=np.stack(chosen), accepted=np.stack(accepted))
    if state["kind"] == "argmax":
        if state["static"]:
            return binding.vocab_argmax_static(state["x"], state["emb"], state["out"])
        return binding.vocab_argmax(state["x"], state["emb"])
    return binding.linear(state["x"], state["W"], state["bias"])


# ------------------------------------------------------------------------------------------------------
# what a pass cannot do without, and how far correct results may lie apart
# ------------------------------------------------------------------------------------------------------
def _model_sizes(shape):
    d, F = shape.d_model, shape.d_ffn
    enc = shape.n_enc * (4 * d * d + 2 * d * F)
    cross_kv = shape.n_dec * 2 * d * d
    dec = shape.n_dec * (6 * d * d + 2 * d * F)
    return enc, cross_kv, dec, shape.vocab * d


def _decode_work(case, out_len, rounds, drafter, block):
    """Weights read once per pass over them, every position multiplied with them once; keys and values of the sources."""
    shape = MODELS[case["model"]]
    s = 2 if shape.dtype == "bf16" else 4
    d, B = shape.d_model, case["batch"]
    enc, ckv, dec, vocab = _model_sizes(shape)
    mean_src = 0.5 * (case["src_lo"] + case["src_hi"])
    models = 2 if drafter else 1
    kv = 2 * shape.n_dec * d * s * B * (mean_src + 0.5 * out_len)
    nbytes = models * s * (enc + ckv) + rounds * (models * (s * (dec + vocab) + kv))
    fed = B * rounds * block
    flops = models * 2 * (enc + ckv) * B * mean_src + 2 * (dec + vocab) * fed
    if drafter:
        flops += 2 * dec * B * rounds * (0.5 * out_len + block) + 2 * vocab * fed
    return {"bytes": float(nbytes), "flops": float(flops)}


def work(case):
    if case["kind"] == "generate":
        T = _max_tgt(case) if case["max_out"] else 0.5 * (case["src_lo"] + case["src_hi"])
        k = min(case["k"], T)
        if k <= 1:
            rounds, block = T, 1.0
        elif case["mode"] == "IAD":           # a rewritten token ends a block and costs a one-token round before the next match
            rounds = max(T / k, 1.0) + 2 * EDIT_RATE * T
            block = 0.5 * (1.0 + min(k, 0.5 * T))
        else:                                 # expected accepted length of a block: a geometric sum
            a = DRAFT_AGREEMENT if case["mode"] == "GAD" else 0.95
            rounds = T / ((1 - a ** k) / (1 - a))
            block = k
        return _decode_work(case, T, max(1.0, rounds), case["mode"] == "GAD", block)
    if case["kind"] == "steps":
        k = min(case["k"], case["src_hi"])
        return _decode_work(case, min(case["src_hi"], 3 * k), STEP_ROUNDS, case["drafter"], 0.5 * k)
    s = 2 if case["dtype"] == "bf16" else 4
    M = case["rows"]
    if case["kind"] == "argmax":
        return {"bytes": float(s * (M + case["vocab"]) * case["d"] + 4 * M), "flops": 2.0 * M * case["vocab"] * case["d"]}
    K, N = case["k_in"], case["n_out"]
    return {"bytes": float(s * (M * K + N * K) + 4 * M * N + 4 * N), "flops": 2.0 * M * N * K}


def tolerance(case):
    if case["kind"] == "linear":
        return {"rel": 1e-5}                  # FP32 sums (BF16 products are exact in FP32)
    if case["kind"] == "argmax":
        return {"rel": 0.0, "differ": 0.002}  # two scores that are equal up to the rounding of FP32 sums
    # token ids: the gaps between the two best scores are far above the rounding of either data type
    return "exact" if MODELS[case["model"]].dtype == "fp32" else {"rel": 0.0, "differ": 0.005}
