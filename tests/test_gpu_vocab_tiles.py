"""Projection + arg-max at the edges of its tiles: 128-token tiles with the tokens on the MMA's M side (65 to 128 tokens), and the
paired kernel's ranges (single 128-row steps where a CTA's range or the vocabulary ends, token tiles that change inside a
range), against a plain FP32 product; equal scores go to the lowest id."""
import numpy as np
import pytest
import torch

from paper_2205_10350_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("M,d,V", [(65, 768, 18945), (100, 1024, 19000), (128, 512, 18944), (127, 256, 50265), (129, 512, 19073),
                                   (257, 448, 10001), (300, 512, 32000), (600, 512, 32000), (1025, 128, 5121), (385, 64, 12672),
                                   (129, 768, 19073), (300, 1024, 13000), (1025, 832, 5121)])
def test_argmax_tiles(M, d, V):
    g = torch.Generator(DEV).manual_seed(M + V)
    x = torch.randn((M, d), generator=g, device=DEV).bfloat16()
    W = torch.randn((V, d), generator=g, device=DEV).bfloat16()
    twins = [(0, 5, V - 1), (M // 2, V // 2, V - 2), (M - 1, 127, 128), (min(M - 1, 64), 255, 256)]
    for m, lo, hi in twins:                   # the same row twice, in different tiles, and the token that likes it best
        W[hi] = W[lo]
        x[m] = (2 * W[lo].float()).bfloat16()
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    got = binding.vocab_argmax(x, W, st).cpu().numpy()
    ref = (x.float() @ W.float().T)
    top, ids = ref.topk(2, 1)
    clear = ((top[:, 0] - top[:, 1]) > 1e-2).cpu().numpy()
    assert np.array_equal(got[clear], ids[:, 0].cpu().numpy()[clear])
    for m, lo in {m: lo for m, lo, _ in twins}.items():
        assert got[m] == lo
    assert clear.sum() > 0.8 * M - 8 and int(st.item()) == 0
