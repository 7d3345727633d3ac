"""Passes of few tokens (register-resident projections, attention with both projections in one kernel, loop planning in the
accept kernel) against the checker, at the edges of their ranges: widths (one to four K chunks, one CTA or a pair per head),
query tiles of 16, rounds of 64 and 32 tokens, the last pass size they take, keys beyond one round of the warps."""
import numpy as np
import pytest

from oracle import ad_oracle as O
from paper_2205_10350_b200 import synth
from tests.parity_util import lockstep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,ffn,batch,k,src,tgt", [
    (256, 512, 1, 1, 3, 9),          # one token
    (256, 768, 2, 17, 66, 70),       # one K chunk, a query tile and one more; keys in two rounds of four warps
    (512, 2048, 1, 64, 40, 128),     # one full round of tokens, last key of the only round
    (512, 1024, 2, 64, 129, 64),     # 128 tokens; source keys in a second round of eight warps
    (512, 512, 1, 33, 20, 129),      # self-attention keys in a second round
    (768, 1536, 3, 9, 30, 24),       # three K chunks, a pair of CTAs with six warps each
    (1024, 1024, 2, 33, 17, 40),     # four K chunks, a pair of CTAs with eight warps each
    (768, 768, 1, 64, 110, 128),     # a pair of CTAs: source keys, then self-attention keys beyond one round of six warps
    (1024, 512, 1, 64, 140, 150),    # the same with eight warps
    (384, 768, 2, 17, 100, 24),      # six warps in one CTA, source keys in a second round
    (640, 640, 1, 20, 90, 24),       # a pair of CTAs with five warps each, source keys in a second round
    (896, 896, 2, 9, 20, 24),        # a pair of CTAs with seven warps each
])
def test_few_token_passes_follow_the_checker(d, ffn, batch, k, src, tgt):
    from paper_2205_10350_b200 import binding
    shape = synth.ModelShape(f"few_{d}_{ffn}", d, d // 64, ffn, 1003, 1, 2, "bf16")
    w = synth.make_weights(shape, 0)
    model = O.Model(shape, w, max_pos=256)
    r = np.random.default_rng(d + batch + k)
    lens = r.integers(max(1, src - 3), src + 1, size=batch).astype(np.int32)
    lens[0] = src
    srcs = r.integers(4, shape.vocab, size=(batch, src)).astype(np.int32)
    dec = binding.AggressiveDecoder(shape, w, max_batch=batch, max_src=src, max_tgt=tgt, kmax=k)
    streams = []
    for b in range(batch):
        g, _ = model.state(srcs[b, : lens[b]], cap=tgt).greedy(tgt)
        row = np.full((1, tgt), 5, np.int32)
        row[0, : len(g)] = g
        streams.append(synth.corrupt_stream(row, [tgt], 0.95, shape.vocab, 9, b)[0])
    stats = lockstep(dec, model, srcs, lens, streams, k, [tgt] * batch, tol=5e-2, max_steps=6)
    print(stats)
    assert stats["steps"] > 0
    dec.close()


def test_vocabulary_as_large_as_the_feed_forward_width():
    """The projection onto the vocabulary and FFN1 share (N, K) in one verification pass and have different launch rules."""
    from paper_2205_10350_b200 import binding
    shape = synth.ModelShape("few_same_width", 256, 4, 1024, 1024, 1, 2, "bf16")
    w = synth.make_weights(shape, 0)
    model = O.Model(shape, w, max_pos=64)
    src = np.random.default_rng(3).integers(4, shape.vocab, size=(3, 11)).astype(np.int32)
    lens = np.array([11, 7, 10], np.int32)
    for k in (50, 33, 7):                    # 150, 99 and 21 tokens of a capacity of 150
        dec = binding.AggressiveDecoder(shape, w, max_batch=3, max_src=11, max_tgt=50, kmax=50)
        streams = [np.resize(model.state(src[b, : lens[b]], cap=50).greedy(50)[0], 50).astype(np.int32) for b in range(3)]
        stats = lockstep(dec, model, src, lens, streams, k, [50] * 3, tol=5e-2, max_steps=2)
        assert stats["steps"] > 0
        dec.close()


@pytest.mark.parametrize("mode,run_drafter,k", [("IAD", False, 7), ("IAD", False, 1), ("GAD", True, 5), ("GAD", True, 12)])
def test_loop_planned_by_the_accept_kernel_equals_one_kernel_per_plan(mode, run_drafter, k, monkeypatch):
    """Whole loops of a ragged batch: planning inside the accept kernel and planning in kernels of their own give the same
    tokens and the same counts, as a graph and as direct launches."""
    from paper_2205_10350_b200 import binding
    shape = synth.MINI_BF16
    w, wn = synth.make_weights(shape, 0), synth.make_weights(shape, 1)
    r = np.random.default_rng(k)
    lens = np.array([12, 5, 1, 9, 12], np.int32)
    src = r.integers(4, 60, size=(5, 12)).astype(np.int32)      # few ids: suffix matches that need more than one token
    results = []
    for env in ("0", "1"):
        monkeypatch.setenv("AD_NO_FUSED_PLAN", env)
        dec = binding.AggressiveDecoder(shape, w, wn if run_drafter else None, max_batch=5, max_src=12, max_tgt=16, kmax=12)
        for graph in (True, False):
            out, st = dec.generate(src, lens, mode=mode, k=k, max_len=[16, 3, 9, 16, 1], run_drafter=run_drafter, use_graph=graph)
            results.append(([list(map(int, o)) for o in out], st["iterations"], st["row_iterations"], st["accepted"], st["offered"]))
        dec.close()
    assert all(x == results[0] for x in results[1:])


@pytest.mark.parametrize("d,batch,k,src", [(256, 2, 17, 129), (256, 1, 5, 192), (512, 1, 16, 257), (512, 2, 9, 400), (768, 1, 17, 200), (1024, 1, 3, 512)])
def test_source_keys_in_three_and_four_rounds(d, batch, k, src):
    """Cross-attention over so many keys that a warp has three or four rounds of them: first and last key count of a round, ragged rows of
    which one ends in the first round."""
    from paper_2205_10350_b200 import binding
    shape = synth.ModelShape(f"rounds_{d}", d, d // 64, 512, 1003, 1, 1, "bf16")
    w = synth.make_weights(shape, 0)
    model = O.Model(shape, w, max_pos=512)
    r = np.random.default_rng(d + src)
    lens = np.array([src, 7][:batch], np.int32)
    srcs = r.integers(4, shape.vocab, size=(batch, src)).astype(np.int32)
    dec = binding.AggressiveDecoder(shape, w, max_batch=batch, max_src=src, max_tgt=k, kmax=k)
    streams = [r.integers(4, shape.vocab, size=k).astype(np.int32) for _ in range(batch)]
    stats = lockstep(dec, model, srcs, lens, streams, k, [k] * batch, tol=5e-2, max_steps=3)
    assert stats["steps"] > 0
    dec.close()


def _needle_model(d):
    """One layer whose self-attention drops everything else for one token, wherever that token is visible."""
    shape = synth.ModelShape(f"needle_{d}", d, d // 64, 512, 1003, 1, 1, "bf16")
    w = synth.make_weights(shape, 0)
    needle, feature = 77, 5
    w["emb"][:, feature] = 0.0
    w["emb"][needle, feature] = 16.0 / np.sqrt(d)             # 16 once scaled; the positional part adds at most 1
    p = "dec.0.self"
    w[f"{p}.o.W"] = synth.round_to_bf16(w[f"{p}.o.W"] * 10.0)
    for h in range(shape.n_heads):
        w[f"{p}.k.W"][feature, h * 64 + 7] = 1.0
        w[f"{p}.q.b"][h * 64 + 7] = 4.0                       # score 8 against at most 0.5 or so: 0.9 of the weight among 400 keys
        w[f"{p}.v.W"][feature, h * 64 + 9: h * 64 + 17] = 0.5
    w["emb"] = synth.round_to_bf16(w["emb"])
    return shape, w, needle


def _blocks(T, k):
    return [(i, min(k, T - i)) for i in range(0, T, k)]


@pytest.mark.parametrize("d,T,k,keys", [(256, 200, 17, (15, 16, 63, 64, 65, 80, 127, 128, 129, 191, 192, 198)),
                                        (256, 180, 9, (64, 112, 128, 176)), (512, 400, 33, (127, 128, 255, 256, 271, 383, 384, 398))])
def test_verified_blocks_see_their_own_keys_in_three_and_four_rounds(d, T, k, keys):
    """Self-attention of blocks over a prefix that reaches three and four rounds of keys per warp, every query with its own number of them:
    a token that takes the whole attention sits on either side of the first key of a warp and of a round, so a query that saw one key
    too many or too few there would choose among other scores altogether."""
    from paper_2205_10350_b200 import binding
    shape, w, needle = _needle_model(d)
    model = O.Model(shape, w, max_pos=512)
    r = np.random.default_rng(d + k)
    src = r.integers(100, shape.vocab, size=(1, 9)).astype(np.int32)
    dec = binding.AggressiveDecoder(shape, w, max_batch=1, max_src=9, max_tgt=T, kmax=k)
    st = model.state(src[0], cap=T)
    for key in keys:
        toks = r.integers(100, shape.vocab, size=T).astype(np.int32)
        toks[key - 1] = needle                                # (key 0 is [BOS])
        st.reset()
        dec.encode(src, [9])
        last = model.bos
        for at, n in _blocks(T, k):
            want = st.verify_block(last, toks[at: at + n], want_logits=True)["logits"]
            dec.verify_block(toks[None, at: at + n], [n])
            err = np.abs(dec.debug_logits(n) - want).max(1)
            assert err.max() <= 5e-2, f"token at key {key}, block from {at}: scores differ by {err.max():.3f} at query {int(err.argmax())}"
            st.commit(n)
            dec.force_commit(toks[None, at: at + n], [n])
            last = int(toks[at + n - 1])
    dec.close()


@pytest.mark.parametrize("d,batch,k,src,rows", [
    (512, 23, 1, 20, (0, 9, 22)),       # an item a row, more items than groups of CTAs by a handful
    (512, 10, 33, 130, (0, 4, 9)),      # three items a row of which some are short, source keys in two rounds
    (512, 40, 1, 260, (0, 31, 32, 39)), # more rows than lanes; source keys in three rounds
    (384, 35, 2, 10, (0, 17, 34)),      # six warps; the last lane's share of the rows is not full
    (768, 4, 33, 100, (0, 1, 3)),       # pairs of CTAs whose halves of the queries meet once an item, keys in two rounds
    (1024, 3, 40, 300, (0, 2)),         # the same with keys in three rounds
])
def test_grids_that_loop_over_the_queries_follow_the_checker(d, batch, k, src, rows, most=None):
    """Attention of passes with more pieces of 16 queries than the device holds CTAs: one verified block of a ragged batch, idle rows among
    the others, at an empty prefix and behind a committed one; sampled rows against the checker.  Blocks of at most `most` tokens (None: k)."""
    most = most or k
    from paper_2205_10350_b200 import binding
    shape = synth.ModelShape(f"loop_{d}", d, d // 64, 512, 1003, 1, 2, "bf16")
    w = synth.make_weights(shape, 0)
    model = O.Model(shape, w, max_pos=320)
    r = np.random.default_rng(d + batch + k)
    lens = r.integers(max(1, src // 3), src + 1, size=batch).astype(np.int32)
    lens[rows[-1]] = src
    srcs = r.integers(4, shape.vocab, size=(batch, src)).astype(np.int32)
    dec = binding.AggressiveDecoder(shape, w, max_batch=batch, max_src=src, max_tgt=2 * k + 1, kmax=k)
    dec.encode(srcs, lens)
    states = {b: model.state(srcs[b, : lens[b]], cap=2 * k + 1) for b in rows}
    last = {b: model.bos for b in rows}
    for turn in range(2):
        drafts = r.integers(4, shape.vocab, size=(batch, k)).astype(np.int32)
        n = np.where(r.random(batch) < 0.2, 0, r.integers(1, most + 1, size=batch)).astype(np.int32)
        n[list(rows)] = [most] + [max(1, most - 5)] * (len(rows) - 2) + [most]
        dec.verify_block(drafts, n)
        lg = dec.debug_logits(int(n.sum()))
        off = np.concatenate([[0], np.cumsum(n)])
        for b in rows:
            want = states[b].verify_block(last[b], drafts[b, : n[b]], want_logits=True)["logits"]
            err = np.abs(lg[off[b]: off[b + 1]] - want).max()
            assert err <= 5e-2, f"row {b}, turn {turn}: scores differ by {err:.3f}"
            states[b].commit(int(n[b]))
            last[b] = int(drafts[b, n[b] - 1])
        dec.force_commit(drafts, n)
    dec.close()


@pytest.mark.parametrize("d,batch,k,src,rows,most", [
    (512, 14, 64, 20, (0, 6, 13), 4),   # a layout for 64 tokens: fewer items than groups, long blocks are possible
    (768, 9, 48, 70, (0, 8), 10),       # the same for 96 tokens and pairs of CTAs
    (768, 13, 18, 70, (0, 7, 12), 4),   # too many items for it: the MMA kernel, few queries in a grid for long blocks
    (1024, 13, 64, 100, (0, 12), 7),    # the same, keys in two tiles
    (768, 24, 64, 70, (0, 11, 23), 1),  # a query a row
])
def test_grids_that_loop_in_layouts_for_few_tokens_follow_the_checker(d, batch, k, src, rows, most):
    test_grids_that_loop_over_the_queries_follow_the_checker(d, batch, k, src, rows, most)


@pytest.mark.parametrize("d,ffn,batch,k", [
    (128, 64, 1, 3),         # one slice of hidden features, two warps
    (256, 1024, 3, 5),       # 16 partial sums, 15 tokens: less than a tile
    (256, 2048, 1, 17),      # 32 partial sums, a tile and one token
    (384, 1536, 2, 40),      # 24 partial sums, six warps; five tiles
    (512, 1088, 2, 64),      # 17 partial sums; eight tiles of tokens, a CTA each
    (512, 2048, 2, 64),      # 32 partial sums; eight tiles for four groups of CTAs
    (512, 2048, 3, 53),      # ten tiles for four groups, the last one short; 160 tokens are the most that 32 partial sums allow
    (384, 1536, 4, 37),      # ten tiles for six groups
])
def test_feed_forward_sublayer_in_one_kernel_follows_the_checker(d, ffn, batch, k):
    test_few_token_passes_follow_the_checker(d, ffn, batch, k, 9, k + 8)
