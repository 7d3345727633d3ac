"""Probabilities of a verification pass's attention keep FP32's weight in passes that are within three waves of the few-query kernel at capacity,
whichever kernel runs them: that one where the tokens are not known when the pass is launched (device arrays), the MMA kernel where they are and are many.

One decoder layer whose scores are dominated by its self-attention or by its cross-attention (wide scores, large values, the other attention and
the feed-forward sublayer without a share) is compared with a float64 restatement that rounds to BF16 only where the model stores an operand:
normalised inputs, queries, keys, values, the attention's output, the hidden states that are scored; the encoder's memory is the library's.  The library may store
a neighbouring BF16 number where an FP32 sum ends near a tie."""
import math

import numpy as np
import pytest
import torch

from paper_2205_10350_b200 import binding, synth

pytestmark = pytest.mark.gpu

BAR = 0.4


def _weights(shape, which):
    w = synth.make_weights(shape, 0)
    for n in list(w):
        if n.startswith(f"dec.0.{which}.") and n.endswith(".W"):
            w[n] = synth.round_to_bf16(w[n] * (6.0 if n.endswith(".o.W") else 3.0))
    other = "cross" if which == "self" else "self"
    for n in (f"dec.0.{other}.o.W", "dec.0.ffn2.W"):
        w[n] = np.zeros_like(w[n])
    return w


def _scores(w, tok, memory, heads, rounded):
    """Scores of one row's first block, whose input tokens are tok, in float64; rounded: stored operands as BF16."""
    d, n = w["emb"].shape[1], len(tok)
    r = (lambda a: synth.round_to_bf16(a.astype(np.float32)).astype(np.float64)) if rounded else (lambda a: a)
    W = {k[len("dec.0."):]: a.astype(np.float64) for k, a in w.items() if k.startswith("dec.0.")}

    def norm(t, nm):
        c = t - t.mean(-1, keepdims=True)
        return W[nm + ".g"] * c / np.sqrt((c ** 2).mean(-1, keepdims=True) + 1e-5) + W[nm + ".b"]

    def attend(x, kv, nm, causal):
        q = r(x @ W[f"{nm}.q.W"] + W[f"{nm}.q.b"])
        k, v = (r(kv @ W[f"{nm}.{c}.W"] + W[f"{nm}.{c}.b"]) for c in "kv")
        q, k, v = (a.reshape(len(a), heads, -1).transpose(1, 0, 2) for a in (q, k, v))
        s = q @ k.transpose(0, 2, 1) / math.sqrt(d // heads)
        if causal:
            s = np.where(np.tril(np.ones((n, n), bool)), s, -np.inf)
        p = np.exp(s - s.max(-1, keepdims=True))
        a = r(((p / p.sum(-1, keepdims=True)) @ v).transpose(1, 0, 2).reshape(n, d))
        return a @ W[f"{nm}.o.W"] + W[f"{nm}.o.b"]

    angle = np.arange(n)[:, None] / 10000.0 ** (np.arange(0, d, 2) / d)[None, :]
    y = w["emb"][tok].astype(np.float64) * math.sqrt(d)
    y[:, 0::2] += np.sin(angle)
    y[:, 1::2] += np.cos(angle)
    x = r(y)
    y = norm(y + attend(x, x, "self", True), "ln1")
    y = norm(y + attend(r(y), memory, "cross", False), "ln2")
    return r(norm(y + W["ffn2.b"], "ln3")) @ w["emb"].astype(np.float64).T


# between two and a half and three waves of CTAs at capacity (148 SMs): 47 to 55 pieces of 16 queries at eight heads, 62 to 74 at six; source keys in one and
# in three rounds; 768 wide between three and four: 19 to 24 pieces
@pytest.mark.parametrize("which", ["self", "cross"])
@pytest.mark.parametrize("d,B,k,S", [(512, 12, 64, 60), (512, 16, 40, 30), (512, 25, 25, 60), (384, 17, 60, 60), (512, 12, 60, 300), (768, 11, 30, 60),
                                       (768, 20, 10, 60)])
def test_verified_blocks_round_only_where_operands_are_stored(d, B, k, S, which):
    shape = synth.ModelShape(f"precision_{d}", d, d // 64, 128, 1003, 1, 1, "bf16")
    w = _weights(shape, which)
    rng = np.random.default_rng(B * 1000 + k)
    src = rng.integers(4, shape.vocab, size=(B, S)).astype(np.int32)
    lens = np.maximum(1, S - 2 * np.arange(B)).astype(np.int32)
    drafts = rng.integers(4, shape.vocab, size=(B, k)).astype(np.int32)
    ks = np.full(B, k, np.int32)
    dec = binding.AggressiveDecoder(shape, w, max_batch=B, max_src=S, max_tgt=k, kmax=k)
    dec.encode(src, lens)
    rows = range(min(B, 3))
    want = []
    for b in rows:
        tok, mem = np.concatenate([[synth.BOS], drafts[b, :-1]]), dec.debug_encoder_memory(b, int(lens[b])).astype(np.float64)
        want.append([_scores(w, tok, mem, shape.n_heads, rounded) for rounded in (True, False)])

    def deviation():
        lg = dec.debug_logits(int(ks.sum()))
        dev = own = 0.0
        for b in rows:
            dev += ((lg[b * k: (b + 1) * k] - want[b][0]) ** 2).sum()
            own += ((want[b][0] - want[b][1]) ** 2).sum()
        return math.sqrt(dev / own)

    ids, n = dec.verify_block(drafts, ks)
    host = deviation()
    t = [torch.tensor(a, device="cuda:0") for a in (drafts, ks, np.zeros_like(drafts), np.zeros_like(ks))]
    dec.verify_block_device(*t)
    dec.sync()
    device = deviation()
    dec.close()
    print(f"{which} {d} wide {B} x {k}, {S} source tokens: deviation {host:.3f} (host arrays), {device:.3f} (device arrays) of the restatement's own")
    assert max(host, device) <= BAR
