"""Captured graphs of a handle: what a program changes from call to call (block-size caps, widths of the draft stream, beta and tau)
does not make the handle capture another one, and reaches calls that replay a graph just as it reaches direct launches."""
import numpy as np
import pytest
import torch

from paper_2205_10350_b200 import binding, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SHAPE = synth.MINI_BF16
B, K, T = 3, 8, 20


def make(monkeypatch=None, **kw):
    if monkeypatch is not None:
        monkeypatch.setenv("AD_NO_ENCODE_GRAPH", "1")       # read when a handle is created: direct launches
    args = dict(max_batch=B, max_src=12, max_tgt=T, kmax=K)
    args.update(kw)
    dec = binding.AggressiveDecoder(SHAPE, synth.make_weights(SHAPE, 0), synth.make_weights(SHAPE, 1), **args)
    if monkeypatch is not None:
        monkeypatch.delenv("AD_NO_ENCODE_GRAPH")
    return dec


def sources(seed=0):
    r = np.random.default_rng(seed)
    return r.integers(4, SHAPE.vocab, size=(B, 12)).astype(np.int32), np.array([12, 5, 9], np.int32)


def test_block_calls_with_changing_settings(monkeypatch):
    graph, direct = make(), make(monkeypatch)
    src, lens = sources()
    r = np.random.default_rng(1)
    counts = []
    for dec in (graph, direct):
        dec.encode(src, lens)
    for step in range(16):
        k_cap = 1 + step % K
        beta, tau = [(0, 0.0), (1, 0.0), (3, 0.5), (40, 2.0 + step)][step // 2 % 4]
        got = []
        drafts = None
        for dec in (graph, direct):
            d, k = dec.draft_block(k_cap)
            if drafts is None:
                assert (k <= k_cap).all()
                drafts, ks = d.copy(), k.copy()
                noise = r.random(d.shape) < 0.3
                drafts[noise] = r.integers(4, SHAPE.vocab, size=int(noise.sum()))
            dec.set_acceptance(beta, tau)
            ids, n = dec.verify_block(drafts, ks)
            take = np.minimum(n, 1)
            dec.commit(take)
            got.append((d, k, ids, n, *dec.state()))
        for a, b in zip(*got):
            assert np.array_equal(a, b), step
        counts.append(graph.debug_graph_count())
    assert direct.debug_graph_count() == 0
    # (exact and relaxed verification are two graphs; every form has run by the fourth step)
    assert counts[-1] == counts[6] <= 4, counts
    graph.close(), direct.close()


def test_whole_calls_with_changing_settings():
    dec = make()
    src, lens = sources(2)
    r = np.random.default_rng(3)
    fresh = {}
    counts = []
    for rnd in range(2):                     # (the second round repeats the first: settings come back)
        for i, (k, width, beta, tau) in enumerate([(8, 20, 0, 0.0), (3, 20, 0, 0.0), (1, 7, 0, 0.0), (5, 11, 2, 0.3), (8, 11, 5, 1.5), (5, 40, 5, 0.1)]):
            stream = np.random.default_rng(i).integers(4, SHAPE.vocab, size=(B, width)).astype(np.int32)
            dec.set_acceptance(beta, tau)
            for mode, drafter, ovr in (("IAD", False, None), ("IAD", False, stream), ("GAD", True, None), ("GAD", True, stream)):
                out, st = dec.generate(src, lens, mode=mode, k=k, max_len=[T, 4, 13], draft_override=ovr, run_drafter=drafter)
                res = ([list(map(int, o)) for o in out], st["iterations"], st["accepted"], st["offered"])
                key = (i, mode, ovr is None)
                if key not in fresh:
                    one = make()
                    one.set_acceptance(beta, tau)
                    o, s = one.generate(src, lens, mode=mode, k=k, max_len=[T, 4, 13], draft_override=ovr, run_drafter=drafter, use_graph=False)
                    fresh[key] = ([list(map(int, a)) for a in o], s["iterations"], s["accepted"], s["offered"])
                    one.close()
                assert res == fresh[key], key
        counts.append(dec.debug_graph_count())
    assert counts[0] == counts[1] <= 8, counts       # four forms, exact and relaxed
    dec.close()


def test_a_form_that_is_called_once_is_not_captured():
    dec = make()
    src, lens = sources(9)
    r = np.random.default_rng(9)
    drafts = r.integers(4, SHAPE.vocab, size=(B, K)).astype(np.int32)
    results = []
    for calls, graphs in ((1, 0), (2, 3), (3, 3)):       # encode, draft, verify
        dec.encode(src, lens)
        d, k = dec.draft_block(5)
        ids, n = dec.verify_block(drafts, [K, 2, 4])
        results.append((d[:, :5].tolist(), k.tolist(), [ids[b, :c].tolist() for b, c in enumerate((K, 2, 4))], n.tolist()))
        assert dec.debug_graph_count() == graphs, calls
    assert results[1] == results[0] and results[2] == results[0]
    dec.close()


def test_captured_graphs_are_bounded():
    """More forms of whole calls than a handle of two rows keeps graphs for: the oldest go, and come back when they are called again."""
    cap = 4 * 2 + 16
    dec = make(max_batch=2)
    src, lens = sources(10)
    stream = np.random.default_rng(11).integers(4, SHAPE.vocab, size=(B, 9)).astype(np.int32)
    first = {}
    for rnd in range(2):
        for rows in (1, 2):
            for relaxed in (0, 2):
                dec.set_acceptance(relaxed, 0.5 if relaxed else 0.0)
                for mode, drafter, ovr in (("IAD", False, None), ("IAD", False, stream), ("GAD", True, None), ("GAD", True, stream), ("GAD", False, stream)):
                    for caps in (None, [7, 9]):
                        out, _ = dec.generate(src[:rows], lens[:rows], mode=mode, k=4, max_len=None if caps is None else caps[:rows],
                                              draft_override=None if ovr is None else ovr[:rows], run_drafter=drafter)
                        key = (rows, relaxed, mode, drafter, ovr is None, caps is None)
                        res = [list(map(int, o)) for o in out]
                        assert first.setdefault(key, res) == res, key
                        assert dec.debug_graph_count() <= cap
    assert len(first) == 40 and dec.debug_graph_count() == cap
    dec.close()


def test_switches_belong_to_the_handle(monkeypatch):
    """A handle made with other switches in the environment does not change what an older one does: one plans its passes in kernels
    of their own, the other in its accept kernel."""
    src, lens = sources(12)
    runs = []
    handles = []
    for own_kernels in ("0", "1"):
        monkeypatch.setenv("AD_NO_FUSED_PLAN", own_kernels)
        handles.append(make())
        runs.append([(st["kernel_launches"], st["iterations"], [list(map(int, o)) for o in out]) for out, st in
                     [h.generate(src, lens, mode="IAD", k=6, max_len=[T, 8, 13], use_graph=False) for h in handles]])
    assert runs[0][0] == runs[1][0]                       # the first handle, before and after the second was made
    assert runs[1][0][1:] == runs[1][1][1:] and runs[1][0][0] < runs[1][1][0]
    for h in handles:
        h.close()


def test_settings_reach_calls_with_device_arrays_in_the_order_they_were_made():
    """Calls with device arrays do not wait: each sees the acceptance rule that was set when it was made."""
    dec, one = make(), make()
    src, lens = sources(4)
    r = np.random.default_rng(5)
    drafts = r.integers(4, SHAPE.vocab, size=(B, K)).astype(np.int32)
    dec.encode(src, lens), one.encode(src, lens)
    d_t, k_t = torch.tensor(drafts, device=DEV), torch.tensor([K, 3, 5], dtype=torch.int32, device=DEV)
    settings = [(0, 0.0), (2000, 1e30), (1, 0.0), (2000, 0.05), (2000, 1e30), (3, 0.4)] * 2
    outs = []
    torch.cuda.synchronize()
    for beta, tau in settings:
        dec.set_acceptance(beta, tau)
        a, n = torch.zeros((B, K), dtype=torch.int32, device=DEV), torch.zeros(B, dtype=torch.int32, device=DEV)
        torch.cuda.synchronize()
        outs.append((a, n))
    for (beta, tau), (a, n) in zip(settings, outs):
        dec.set_acceptance(beta, tau)
        dec.verify_block_device(d_t, k_t, a, n)
    dec.sync()
    seen = set()
    for (beta, tau), (a, n) in zip(settings, outs):
        one.set_acceptance(beta, tau)
        ids, m = one.verify_block(drafts, [K, 3, 5])
        for b, k in enumerate((K, 3, 5)):
            assert np.array_equal(a[b, :k].cpu().numpy(), ids[b, :k])
        assert np.array_equal(n.cpu().numpy(), m)
        seen.add(tuple(m))
    assert len(seen) > 1
    dec.close(), one.close()


def test_block_size_caps_of_draft_calls_with_device_arrays():
    dec, one = make(), make()
    src, lens = sources(8)
    dec.encode(src, lens), one.encode(src, lens)
    caps = [1, K, 3, 5, 5, 2] * 2
    outs = [(torch.zeros((B, K), dtype=torch.int32, device=DEV), torch.zeros(B, dtype=torch.int32, device=DEV)) for _ in caps]
    torch.cuda.synchronize()
    for cap, (d, k) in zip(caps, outs):
        assert dec.lib.ad_draft_block(dec.h, cap, d.data_ptr(), k.data_ptr(), 0) == binding.AD_OK
    dec.sync()
    for cap, (d, k) in zip(caps, outs):
        d1, k1 = one.draft_block(cap)
        assert np.array_equal(k.cpu().numpy(), k1) and (k1 == cap).all()
        assert np.array_equal(d[:, :cap].cpu().numpy(), d1[:, :cap])
    assert dec.debug_graph_count() <= 2
    dec.close(), one.close()


def test_a_callers_own_graph_keeps_its_settings():
    """A block verified inside a graph that the caller records keeps the rule it was recorded with, and later calls keep theirs."""
    stream = torch.cuda.Stream()
    dec = make(stream=stream)
    src, lens = sources(6)
    drafts = np.random.default_rng(7).integers(4, SHAPE.vocab, size=(B, K)).astype(np.int32)
    d_t, k_t = torch.tensor(drafts, device=DEV), torch.tensor([K, K, K], dtype=torch.int32, device=DEV)
    a, n = torch.zeros((B, K), dtype=torch.int32, device=DEV), torch.zeros(B, dtype=torch.int32, device=DEV)
    dec.encode(src, lens)
    dec.set_acceptance(2000, 1e30)           # keeps every draft
    dec.verify_block(drafts, [K] * B)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        dec.verify_block_device(d_t, k_t, a, n)
    dec.set_acceptance(0, 0.0)
    exact = dec.verify_block(drafts, [K] * B)[1]
    assert (exact < K).any()
    for _ in range(2):
        with torch.cuda.stream(stream):
            g.replay()
        dec.sync()
        assert (n.cpu().numpy() == K).all()
        assert np.array_equal(dec.verify_block(drafts, [K] * B)[1], exact)
    del g
    dec.close()
