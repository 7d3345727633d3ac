"""A property that holds at any size: a row's verified block does not depend on which other rows share its pass.

Batched passes of different sizes take different kernels and launch shapes (token tiles of 32, 64 or 128, split-K
factors, the attention kernel for few queries / many queries / hundreds of keys, the persistent projection kernel), a
single row takes the small-pass ones.  The scores of sampled rows of a ragged batch are compared with the same rows
verified alone; both sides are the library, so this pins no arithmetic -- the checker does that at sizes it can afford
(test_gpu_parity.py) -- but it ties every large-pass configuration to the small-pass path the checker follows
element by element.  Tolerance: the BF16 bar (the two sides differ in summation order only)."""
import numpy as np
import pytest

from oracle import ad_oracle as O
from paper_2205_10350_b200 import binding, synth
from tests.parity_util import following_weights

pytestmark = pytest.mark.gpu

CASES = [("base", synth.BASE, 8, 25, 400),       # 200-token capacity: 32-token tiles, keys spread over warps
         ("base", synth.BASE, 32, 30, 48),       # 960: 64-token tiles, tensor-core attention, persistent projection
         ("big", synth.BIG, 4, 25, 32),          # 100: K loops of several ring rounds
         ("big", synth.BIG, 16, 64, 32),         # 1024
         ("bart", synth.BART_BASE_SIZED, 6, 30, 40),   # 12 heads, K blocks not a power of two
         ("base", synth.BASE, 3, 64, 300)]       # 192: long sources with long blocks


@pytest.mark.parametrize("name,shape,B,k,S", CASES, ids=[f"{c[0]}-{c[2]}x{c[3]}-src{c[4]}" for c in CASES])
def test_batched_pass_agrees_with_single_row_passes(name, shape, B, k, S):
    r = np.random.default_rng(B * 1000 + k)
    w = synth.make_weights(shape, 0)
    src = r.integers(4, shape.vocab, size=(B, S)).astype(np.int32)
    lens = r.integers(max(1, S // 2), S + 1, size=B).astype(np.int32)
    ks = r.integers(1, k + 1, size=B).astype(np.int32)
    ks[B - 1] = k                                         # one full-length block
    drafts = r.integers(4, shape.vocab, size=(B, k)).astype(np.int32)
    dec = binding.AggressiveDecoder(shape, w, max_batch=B, max_src=S, max_tgt=k, kmax=k)
    dec.encode(src, lens)
    ids, n = dec.verify_block(drafts, ks)
    lg = dec.debug_logits(int(ks.sum()))
    dec.close()
    offs = np.concatenate([[0], np.cumsum(ks)])
    one = binding.AggressiveDecoder(shape, w, max_batch=1, max_src=S, max_tgt=k, kmax=k)
    worst = 0.0
    for b in sorted({0, B // 2, B - 1}):
        one.encode(src[b: b + 1], lens[b: b + 1])
        ids1, n1 = one.verify_block(drafts[b: b + 1], ks[b: b + 1])
        l1 = one.debug_logits(int(ks[b]))
        got = lg[offs[b]: offs[b + 1]]
        worst = max(worst, float(np.abs(got - l1).max()))
        # ids agree wherever the single-row scores leave no doubt
        top2 = np.sort(l1, axis=1)[:, -2:]
        clear = (top2[:, 1] - top2[:, 0]) > 0.1
        assert (ids[b, : ks[b]][clear] == ids1[0, : ks[b]][clear]).all()
    one.close()
    print(f"{name} B={B} k={k} S={S}: worst |batched - alone| = {worst:.4f}")
    assert worst <= 5e-2


DRAFT_CASES = [("base", synth.BASE, 8, 25, 400, 40), ("big", synth.BIG, 4, 25, 40, 30), ("mini", synth.MINI_BF16, 6, 16, 30, 200)]


@pytest.mark.parametrize("name,shape,B,k,S,T", DRAFT_CASES, ids=[f"{c[0]}-{c[2]}rows-prefix<={c[5]}" for c in DRAFT_CASES])
def test_batched_drafter_pass_agrees_with_single_row_passes(name, shape, B, k, S, T):
    """The same for the drafter's pass (Section 3.2.1): rows are walked to ragged prefixes by teacher forcing, then the
    draft scores of sampled rows of the batch are compared with the same rows drafted alone."""
    r = np.random.default_rng(B * 100 + T)
    w, wn = synth.make_weights(shape, 0), synth.make_weights(shape, 1)
    src = r.integers(4, shape.vocab, size=(B, S)).astype(np.int32)
    lens = r.integers(max(1, S // 2), S + 1, size=B).astype(np.int32)
    prefixes = [r.integers(4, shape.vocab, size=int(n)).astype(np.int32) for n in r.integers(0, T + 1, size=B)]

    def draft(dec, rows):
        dec.encode(src[rows], lens[rows])
        done = [0] * len(rows)
        while any(done[i] < len(prefixes[b]) for i, b in enumerate(rows)):
            ks = np.zeros(len(rows), np.int32)
            toks = np.full((len(rows), dec.kmax), -1, np.int32)
            for i, b in enumerate(rows):
                seg = prefixes[b][done[i]: done[i] + dec.kmax]
                ks[i] = len(seg)
                toks[i, : len(seg)] = seg
                done[i] += len(seg)
            dec.verify_block(toks, ks)
            dec.force_commit(toks, ks)
        d, kk = dec.draft_block(k)
        return d, kk, dec.debug_logits(int(kk.sum()), which=1)

    dec = binding.AggressiveDecoder(shape, w, wn, max_batch=B, max_src=S, max_tgt=T + k, kmax=k)
    d, kk, scores = draft(dec, list(range(B)))
    dec.close()
    offs = np.concatenate([[0], np.cumsum(kk)])
    one = binding.AggressiveDecoder(shape, w, wn, max_batch=1, max_src=S, max_tgt=T + k, kmax=k)
    worst = 0.0
    for b in sorted({0, B // 2, B - 1}):
        d1, k1, s1 = draft(one, [b])
        assert int(k1[0]) == int(kk[b])
        worst = max(worst, float(np.abs(scores[offs[b]: offs[b + 1]] - s1).max()))
    one.close()
    print(f"{name} B={B}: drafter worst |batched - alone| = {worst:.4f}")
    assert worst <= 5e-2


LOOP_CASES = [(5, 64, 40, "IAD", False), (8, 25, 100, "GAD", True), (32, 64, 48, "IAD", False), (4, 40, 300, "GAD", True)]


@pytest.mark.parametrize("B,k,S,mode,drafter", LOOP_CASES, ids=[f"{c[3]}-{c[0]}rows-k{c[1]}-src{c[2]}" for c in LOOP_CASES])
def test_decode_loop_as_one_graph_equals_direct_launches_at_every_pass_size(B, k, S, mode, drafter):
    """The whole loop (Algorithm 1 / Section 3.2) on the base model at several batch sizes: one graph launch with the
    device-side loop, the same call again, and direct launches with host polling must return identical tokens and
    iteration counts.  How many rows also equal the library's own greedy decoding (block size 1, other kernels and launch
    shapes) is printed: the method is lossless, so every row whose positions are all clear of near-ties does."""
    shape = synth.BASE
    r = np.random.default_rng(B * 7 + k)
    w = synth.make_weights(shape, 0)
    wn = synth.make_weights(shape, 1) if drafter else None
    T = max(48, k)
    dec = binding.AggressiveDecoder(shape, w, wn, max_batch=B, max_src=S, max_tgt=T, kmax=k)
    src = r.integers(4, shape.vocab, size=(B, S)).astype(np.int32)
    lens = r.integers(max(1, S // 2), S + 1, size=B).astype(np.int32)
    max_len = r.integers(8, T + 1, size=B).astype(np.int32)
    g, _ = dec.generate(src, lens, mode="IAD", k=1, max_len=max_len)
    gg = np.full((B, T), synth.PAD, np.int32)
    for b in range(B):
        gg[b, : len(g[b])] = g[b]
    kw = dict(mode=mode, k=k, max_len=max_len)
    if drafter:
        kw["run_drafter"] = True
    else:
        kw["draft_override"] = synth.corrupt_stream(gg, [len(x) for x in g], 0.8, shape.vocab, 3, B)
    a, sa = dec.generate(src, lens, use_graph=True, **kw)
    d, sd = dec.generate(src, lens, use_graph=False, **kw)
    c, sc = dec.generate(src, lens, use_graph=True, **kw)
    for b in range(B):
        assert np.array_equal(a[b], d[b]) and np.array_equal(a[b], c[b]), b
        assert 1 <= len(a[b]) <= max_len[b]
    assert sa["iterations"] == sd["iterations"] == sc["iterations"]
    same = sum(np.array_equal(a[b], g[b]) for b in range(B))
    print(f"B={B} k={k} S={S} {mode}: {sa['iterations']} iterations, {same}/{B} rows identical to block-size-1 decoding")
    assert same >= B - max(1, B // 4)          # near-ties may move a few rows off; a broken loop moves all of them
    dec.close()


# last and first capacity on either side of the lines between the encoder's attention kernels (148 SMs): few-query to MMA or FFMA kernel, FFMA to
# MMA kernel (more than one key tile, more CTAs), MMA kernel to the same for many queries, and 256 keys and more
ENCODE_CASES = [("base", synth.BASE, 5, 80), ("base", synth.BASE, 5, 81), ("base", synth.BASE, 2, 200), ("base", synth.BASE, 2, 208),
                ("base", synth.BASE, 2, 209), ("base", synth.BASE, 2, 216), ("base", synth.BASE, 2, 217), ("base", synth.BASE, 1, 288),
                ("base", synth.BASE, 1, 289), ("bart", synth.BART_BASE_SIZED, 2, 48), ("bart", synth.BART_BASE_SIZED, 2, 49),
                ("bart", synth.BART_BASE_SIZED, 2, 64), ("bart", synth.BART_BASE_SIZED, 2, 65), ("bart", synth.BART_BASE_SIZED, 2, 97),
                ("bart", synth.BART_BASE_SIZED, 2, 50), ("bart", synth.BART_BASE_SIZED, 2, 144), ("bart", synth.BART_BASE_SIZED, 2, 145),
                ("bart", synth.BART_BASE_SIZED, 9, 16), ("bart", synth.BART_BASE_SIZED, 10, 16), ("bart", synth.BART_BASE_SIZED, 24, 8),
                ("bart", synth.BART_BASE_SIZED, 25, 8), ("big", synth.BIG, 2, 32), ("big", synth.BIG, 2, 33), ("big", synth.BIG, 2, 48),
                ("big", synth.BIG, 2, 49)]


@pytest.mark.parametrize("name,shape,B,S", ENCODE_CASES, ids=[f"{c[0]}-{c[2]}x{c[3]}" for c in ENCODE_CASES])
def test_encoder_rows_agree_with_single_row_passes(name, shape, B, S):
    """The encoder memory of the longest and the shortest row of a ragged batch against the same rows encoded alone (unit-variance rows;
    the bar is the one of the comparison with the checker)."""
    r = np.random.default_rng(B * 1000 + S)
    w = synth.make_weights(shape, 0)
    src = r.integers(4, shape.vocab, size=(B, S)).astype(np.int32)
    lens = r.integers(1, S + 1, size=B).astype(np.int32)
    lens[B - 1] = S
    dec = binding.AggressiveDecoder(shape, w, max_batch=B, max_src=S, max_tgt=4, kmax=4)
    dec.encode(src, lens)
    for b in {int(np.argmin(lens)), B - 1}:
        n = int(lens[b])
        one = binding.AggressiveDecoder(shape, w, max_batch=1, max_src=n, max_tgt=4, kmax=4)
        one.encode(src[b: b + 1, :n], lens[b: b + 1])
        diff = np.abs(dec.debug_encoder_memory(b, n) - one.debug_encoder_memory(0, n)).max()
        one.close()
        assert diff <= 5e-2
    dec.close()


@pytest.mark.parametrize("B", [2, 8, 9, 16, 17])
def test_rows_of_a_loop_end_like_single_rows(B):
    """Decode loops around the numbers of rows whose accept kernels are one cluster (8 CTAs everywhere, up to 16 here, none beyond): tokens,
    iterations and offered drafts of every row as in a loop of its own.  FP32: the arithmetic leaves no doubt."""
    shape = synth.TINY
    w, wn = synth.make_weights(shape, 0), synth.make_weights(shape, 1)
    r = np.random.default_rng(B)
    S, T = 12, 14
    src = r.integers(4, shape.vocab, size=(B, S)).astype(np.int32)
    lens = r.integers(2, S + 1, size=B).astype(np.int32)
    cap = r.integers(1, T + 1, size=B).astype(np.int32)
    many = binding.AggressiveDecoder(shape, w, wn, max_batch=B, max_src=S, max_tgt=T, kmax=6)
    one = binding.AggressiveDecoder(shape, w, wn, max_batch=1, max_src=S, max_tgt=T, kmax=6)
    for opts in (dict(mode="IAD", k=6), dict(mode="GAD", k=5, run_drafter=True)):
        out, st = many.generate(src, lens, max_len=cap, **opts)
        alone = [one.generate(src[b: b + 1], lens[b: b + 1], max_len=cap[b: b + 1], **opts) for b in range(B)]
        assert all(np.array_equal(out[b], alone[b][0][0]) for b in range(B))
        assert st["iterations"] == max(a[1]["iterations"] for a in alone)
        for key in ("row_iterations", "accepted", "offered"):
            assert st[key] == sum(a[1][key] for a in alone)
    many.close()
    one.close()


def _loop_results(dec, src, lens, cap, stream, relaxed):
    runs = [dict(mode="IAD", k=6), dict(mode="GAD", k=5, run_drafter=True), dict(mode="GAD", k=6, draft_override=stream)]
    out = []
    for beta in ((0, 2) if relaxed else (0,)):
        dec.set_acceptance(beta, 0.5)
        for opts in runs:
            rows, st = dec.generate(src, lens, max_len=cap, **opts)
            out.append(([r.tolist() for r in rows], [st[key] for key in ("iterations", "row_iterations", "accepted", "offered")]))
    return out


@pytest.mark.parametrize("B", [2, 7, 8, 9, 16, 17])
def test_rows_of_a_loop_meet_in_a_cluster_or_through_global_memory(B, monkeypatch):
    """BF16 loops with drafts from the source, the drafter and the caller, exact and relaxed: the same tokens and counts whether the rows'
    accept kernels are one cluster as large as the device places it, one of at most eight rows, or meet through global memory as on a
    device that places none."""
    shape = synth.MINI_BF16
    w, wn = synth.make_weights(shape, 0), synth.make_weights(shape, 1)
    r = np.random.default_rng(100 + B)
    S, T = 12, 14
    src = r.integers(4, 60, size=(B, S)).astype(np.int32)
    lens = r.integers(2, S + 1, size=B).astype(np.int32)
    cap = r.integers(1, T + 1, size=B).astype(np.int32)
    stream = r.integers(4, shape.vocab, size=(B, T)).astype(np.int32)
    results = []
    for limit in (None, "8", "0"):
        if limit is not None:
            monkeypatch.setenv("AD_ACCEPT_CLUSTER", limit)      # read when a handle is created
        dec = binding.AggressiveDecoder(shape, w, wn, max_batch=B, max_src=S, max_tgt=T, kmax=6)
        greedy, _ = dec.generate(src, lens, max_len=cap, k=1)
        for b in range(0, B, 2):                                # long accepted blocks in every other row
            stream[b, : len(greedy[b])] = greedy[b]
        results.append(_loop_results(dec, src, lens, cap, stream, relaxed=True))
        dec.close()
    assert results[1] == results[0] and results[2] == results[0]


BODY_CASES = [(512, 5, 13, "stream"), (512, 7, 14, "stream"), (512, 24, 40, "stream"), (512, 33, 9, "policy"), (512, 26, 40, "policy"), (768, 7, 14, "relaxed"),
              (768, 20, 20, "policy"), (512, 5, 20, "drafter")]


@pytest.mark.parametrize("d,B,k,how", BODY_CASES, ids=[f"{c[3]}-{c[0]}wide-{c[1]}rows-k{c[2]}" for c in BODY_CASES])
def test_bodies_of_a_loop_for_few_and_many_tokens_give_the_same_sentences(d, B, k, how, monkeypatch):
    """A decode loop picks its body by the tokens of each iteration; with one body for all of them (and with direct launches) the sentences and the
    iterations are the same but for near-ties, and the launches that are counted are those of the bodies that ran."""
    shape = synth.ModelShape(f"bodies_{d}", d, d // 64, 512, 1003, 1, 2, "bf16")
    w = synth.make_weights(shape, 0)
    wn = synth.make_weights(shape, 1) if how == "drafter" else None
    r = np.random.default_rng(d + B * 7 + k)
    T = max(24, k)
    src = r.integers(4, 200, size=(B, T)).astype(np.int32)
    lens = r.integers(T // 2, T + 1, size=B).astype(np.int32)
    max_len = r.integers(4, T + 1, size=B).astype(np.int32)
    max_len[0] = T
    kw = dict(mode="IAD" if how == "policy" else "GAD", k=k, max_len=max_len)
    if how == "drafter":
        kw["run_drafter"] = True
    elif how != "policy":
        kw["draft_override"] = r.integers(4, shape.vocab, size=(B, T)).astype(np.int32)
    runs = []
    for one_body in ("0", "1"):
        monkeypatch.setenv("AD_NO_FEW_BODY", one_body)
        dec = binding.AggressiveDecoder(shape, w, wn, max_batch=B, max_src=T, max_tgt=T, kmax=k)
        if how == "relaxed":
            dec.set_acceptance(4, 0.5)
        first, a = dec.generate(src, lens, **kw)
        again, b = dec.generate(src, lens, **kw)
        assert all(np.array_equal(x, y) for x, y in zip(first, again)) and a["kernel_launches"] == b["kernel_launches"]
        direct, s = dec.generate(src, lens, use_graph=False, **kw)
        runs += [(first, a), (direct, s)]
        if one_body == "1":
            assert a["kernel_launches"] >= a["iterations"] * 10
        dec.close()
    same = [sum(np.array_equal(x, y) for x, y in zip(runs[0][0], other[0])) for other in runs[1:]]
    print(f"{how} {d} wide B={B} k={k}: rows the same {same}, iterations {[x[1]['iterations'] for x in runs]}, launches {[x[1]['kernel_launches'] for x in runs]}")
    assert min(same) >= B - max(1, B // 4)


# capacities just beyond what one form holds (96 tokens, 128 for the policy) and far beyond
FOLLOWING_CASES = [(512, 7, 14, "stream"), (512, 24, 40, "stream"), (512, 33, 9, "policy"), (512, 10, 13, "policy"), (768, 7, 14, "relaxed"),
              (768, 20, 20, "policy"), (512, 5, 20, "drafter")]
BETA, TAU = 4, 0.5


def _parts_at_a_near_tie(model, src, a, b, draft):
    """Whether two outputs of a row first differ where the checker's scores leave the choice open: the best two close together or, with drafts
    accepted by rank and distance, the draft close to either limit."""
    n = min(len(a), len(b))
    differs = np.nonzero(np.asarray(a[:n]) != np.asarray(b[:n]))[0]
    at = int(differs[0]) if len(differs) else n - 1           # (one ends there: [EOS] was chosen or accepted as the last token of both)
    prefix = [int(t) for t in a[:at]]
    scores = model.state(src, cap=len(prefix) + 1).verify_block(model.bos, prefix + [5], want_logits=True)["logits"][at]
    top = np.sort(scores)[::-1]
    if top[0] - top[1] <= 0.1:
        return True
    if draft is None:
        return False
    d = scores[draft[at]]
    return min(abs(top[0] - d - TAU), abs(top[BETA - 1] - d), abs(top[BETA] - d)) <= 0.1


@pytest.mark.parametrize("d,B,k,how", FOLLOWING_CASES, ids=[f"{c[3]}-{c[0]}wide-{c[1]}rows-k{c[2]}" for c in FOLLOWING_CASES])
def test_bodies_of_a_loop_differ_at_near_ties_alone(d, B, k, how, monkeypatch):
    """A decode loop picks its body by the tokens of each iteration; with one body for all of them and with direct launches the sentences are the
    same or part at a near-tie, and so are the iterations where all sentences are the same and the drafts do not come from the drafter."""
    shape = synth.ModelShape(f"bodies_{d}", d, d // 64, 512, 1003, 1, 2, "bf16")
    w = following_weights(shape)
    wn = synth.make_weights(shape, 1) if how == "drafter" else None
    r = np.random.default_rng(d + B * 7 + k)
    T = max(24, k)
    src = r.integers(4, 200, size=(B, T)).astype(np.int32)
    lens = r.integers(T // 2, T + 1, size=B).astype(np.int32)
    lens[0] = T
    max_len = np.minimum(lens, r.integers(4, T + 1, size=B)).astype(np.int32)
    max_len[0] = T
    kw = dict(mode="IAD" if how == "policy" else "GAD", k=k, max_len=max_len)
    stream = None
    if how == "drafter":
        kw["run_drafter"] = True
    elif how != "policy":
        stream = kw["draft_override"] = np.where(r.random((B, T)) < 0.1, r.integers(4, shape.vocab, size=(B, T)), src).astype(np.int32)
    runs = []
    for one_body in ("0", "1"):
        monkeypatch.setenv("AD_NO_FEW_BODY", one_body)
        dec = binding.AggressiveDecoder(shape, w, wn, max_batch=B, max_src=T, max_tgt=T, kmax=k)
        if how == "relaxed":
            dec.set_acceptance(BETA, TAU)
        first, a = dec.generate(src, lens, **kw)
        again, b = dec.generate(src, lens, **kw)
        assert all(np.array_equal(x, y) for x, y in zip(first, again)) and a["kernel_launches"] == b["kernel_launches"]
        direct, s = dec.generate(src, lens, use_graph=False, **kw)
        runs += [(first, a), (direct, s)]
        dec.close()
    copied = np.mean([np.mean(np.where(src[b, : len(row)] % 8, src[b, : len(row)], src[b, : len(row)] + 1) == row) for b, row in enumerate(runs[0][0])])
    assert copied > 0.6                                       # (the model follows its sources, at low positions by one token more or less)
    model = O.Model(shape, w, max_pos=64)
    for other, stats in runs[1:]:
        parted = [b for b in range(B) if not np.array_equal(runs[0][0][b], other[b])]
        for b in parted:
            assert _parts_at_a_near_tie(model, src[b, : lens[b]], runs[0][0][b], other[b], stream[b] if how == "relaxed" else None), b
        if not parted and how != "drafter":
            assert stats["iterations"] == runs[0][1]["iterations"]
        print(f"{how} {d} wide B={B} k={k}: rows that part {parted}, iterations {runs[0][1]['iterations']} and {stats['iterations']}")


# (width, rows, block size, capacities of the forms): the lines for 148 SMs
FORM_CASES = [(512, 6, 16, (96,)), (512, 7, 14, (64, 98)), (512, 24, 40, (64, 352, 960)), (512, 33, 9, (64, 297)), (768, 20, 20, (96, 400)), (768, 6, 17, (96, 102))]


@pytest.mark.parametrize("d,B,k,caps", FORM_CASES, ids=[f"{c[0]}wide-{c[1]}rows-k{c[2]}" for c in FORM_CASES])
def test_launches_counted_are_those_of_the_forms_that_ran(d, B, k, caps, monkeypatch):
    """Drafts that are never accepted: every iteration adds a token a row, so the tokens of each, and with them the form of the body that
    holds them, are known.  The kernels that a call launched are those of these forms."""
    shape = synth.ModelShape(f"bodies_{d}", d, d // 64, 512, 1003, 1, 2, "bf16")
    w = synth.make_weights(shape, 0)
    r = np.random.default_rng(d + B * 7 + k)
    T = 48
    src = r.integers(4, 200, size=(B, 24)).astype(np.int32)
    lens = r.integers(12, 25, size=B).astype(np.int32)
    max_len = r.integers(T // 2, T + 1, size=B).astype(np.int32)
    max_len[0] = T

    def call(dec, cap, k):
        used = {int(t) for row in dec.generate(src, lens, mode="IAD", k=1, max_len=cap)[0] for t in row}
        stream = np.full((B, T), min(set(range(4, shape.vocab)) - used), np.int32)
        out, st = dec.generate(src, lens, mode="GAD", k=k, max_len=cap, draft_override=stream)
        n = np.array([len(row) for row in out])
        tokens = [int(np.minimum(k, cap - t)[n > t].sum()) for t in range(n.max())]
        assert st["iterations"] == len(tokens) and st["offered"] == sum(tokens), "a draft was accepted"
        return tokens, st["kernel_launches"]

    def per_iteration(dec, k):                                # of a loop that stays in one form, and what it launches outside
        (t1, n1), (t2, n2) = call(dec, np.full(B, 8, np.int32), k), call(dec, np.full(B, 3, np.int32), k)
        each = (n1 - n2) // (len(t1) - len(t2))
        assert n1 - n2 == each * (len(t1) - len(t2))
        return each, n1 - each * len(t1)

    monkeypatch.setenv("AD_NO_FEW_BODY", "1")
    one = binding.AggressiveDecoder(shape, w, max_batch=B, max_src=24, max_tgt=T, kmax=k)
    full, _ = per_iteration(one, k)
    one.close()
    monkeypatch.setenv("AD_NO_FEW_BODY", "0")
    dec = binding.AggressiveDecoder(shape, w, max_batch=B, max_src=24, max_tgt=T, kmax=k)
    few, once = per_iteration(dec, 1)
    # between the two: the embedding as a kernel of its own; the feed-forward sublayer stays in one kernel (512 wide, 8 slices: up to 640 tokens)
    kernels = [few, few + 1, full][: len(caps)]
    if len(caps) == 2 and d > 512:
        # (a handle of 65 to 128 tokens and one form has the embedding in the projection, the last of several forms does not)
        kernels = [few, full + (1 if caps[-1] <= 128 else 0)]
    tokens, launched = call(dec, max_len, k)
    dec.close()
    forms = [sum(t > c for c in caps[:-1]) for t in tokens]
    print(f"{d} wide B={B} k={k}: kernels {kernels}, {full} in one form, iterations {[forms.count(i) for i in range(len(caps))]}")
    assert launched == once + sum(kernels[f] for f in forms)
    assert all(forms.count(i) > 0 for i in range(len(caps)))
