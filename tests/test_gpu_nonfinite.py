"""Scores that are not finite: whatever a model's activations are, a choice is an id of the vocabulary (ids index the embedding
matrix in the next pass), and -inf scores order like any others: equal ones go to the lowest id."""
import numpy as np
import pytest
import torch

from paper_2205_10350_b200 import binding, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype,M,d,V", [("bf16", 7, 128, 1000), ("bf16", 7, 128, 1025), ("bf16", 100, 128, 19000), ("bf16", 300, 512, 19073), ("bf16", 300, 768, 19073),
                                         ("fp32", 5, 64, 1000), ("fp32", 40, 64, 12900), ("fp32", 300, 64, 200)])
def test_argmax_of_infinite_and_nan_scores(dtype, M, d, V):
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(DEV).manual_seed(M)
    x, W = torch.randn((M, d), generator=g, device=DEV).to(dt), torch.randn((V, d), generator=g, device=DEV).to(dt)
    W[:, 0], W[:, 1] = 1.0, 1.0
    W[V - 1, 1] = -1.0
    x[0, 0] = -np.inf                     # every score -inf
    x[1, 1] = -np.inf                     # every score -inf but the last, +inf
    x[2] = np.nan
    got = binding.vocab_argmax(x, W).cpu().numpy()
    assert got[0] == 0 and got[1] == V - 1 and 0 <= got[2] < V
    assert (got >= 0).all() and (got < V).all()


@pytest.mark.parametrize("shape,batch", [(synth.MINI_BF16, 2), (synth.MINI_BF16, 20), (synth.TINY, 2)])
@pytest.mark.parametrize("value", [-np.inf, np.nan])
def test_decode_loops_on_non_finite_scores_stay_inside_the_vocabulary(shape, batch, value):
    """Both models' last LayerNorm gives hidden states whose scores are all -inf or NaN: the loop still feeds tokens that exist."""
    ws = []
    for m in range(2):
        w = {n: a.copy() for n, a in synth.make_weights(shape, m).items()}
        w["emb"][:, 0] = 1.0
        w[f"dec.{shape.n_dec - 1}.ln3.b"][0] = value
        ws.append(w)
    dec = binding.AggressiveDecoder(shape, ws[0], ws[1], max_batch=batch, max_src=12, max_tgt=16, kmax=8)
    r = np.random.default_rng(batch)
    src = r.integers(4, shape.vocab, size=(batch, 12)).astype(np.int32)
    lens = r.integers(1, 13, size=batch).astype(np.int32)
    for mode, drafter in (("IAD", False), ("GAD", True)):
        for graph in (True, False):
            rows, _ = dec.generate(src, lens, mode=mode, k=5, max_len=[10] * batch, run_drafter=drafter, use_graph=graph)
            for out in rows:
                assert (out >= 0).all() and (out < shape.vocab).all()
                if value == -np.inf:
                    assert (out == 0).all() and len(out) == 10     # all scores equal: the lowest id
    dec.encode(src, lens)
    drafts, k = dec.draft_block(5)
    assert (k == 5).all() and (drafts[:, :5] >= 0).all() and (drafts[:, :5] < shape.vocab).all()
    dec.close()
