"""The C-ABI library loads on a machine without a GPU and exports every symbol the header declares;
host-only entry points (sizes, configuration checks) behave."""
import ctypes as C
import os
import re

import pytest

from paper_2205_10350_b200 import binding, build, synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    build.build()
    return binding.load()


def declared_functions():
    text = open(os.path.join(ROOT, "include", "aggressive_decoding.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(ad_[a-z_0-9]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    names = declared_functions()
    assert len(names) >= 15
    for n in names:
        assert hasattr(lib, n), n
    assert sorted(binding.EXPORTS) == names


def _cfg(shape, **kw):
    args = dict(max_batch=1, max_src=40, max_tgt=40, kmax=40)
    args.update(kw)
    return binding.ModelCfg(shape.d_model, shape.n_heads, shape.d_ffn, shape.vocab, shape.n_enc, shape.n_dec,
                            1 if shape.dtype == "bf16" else 0, args["max_batch"], args["max_src"], args["max_tgt"],
                            args["kmax"], 0, 1, 2, 3, 1e-5, args.get("has_drafter", 0))


def test_weight_counts_match_the_documented_layout(lib):
    for shape in (synth.TINY, synth.BASE):
        cfg = _cfg(shape)
        nm, nv = C.c_size_t(), C.c_size_t()
        assert lib.ad_weight_counts(C.byref(cfg), C.byref(nm), C.byref(nv)) == 0
        d, F, V = shape.d_model, shape.d_ffn, shape.vocab
        mats = V * d + shape.n_enc * (4 * d * d + 2 * d * F) + shape.n_dec * (8 * d * d + 2 * d * F)
        assert nm.value == mats
        w = {n: __import__("numpy").zeros(s, "float32") for n, s in synth.weight_names(shape)}
        m, v = binding.pack_weights(shape, w)
        assert (m.size, v.size) == (nm.value, nv.value)
    # per-verify streamed weights of the base model: 6 (6 d^2 + 2 d F) + V d parameters
    d, F, V = 512, 2048, 32000
    assert 6 * (6 * d * d + 2 * d * F) + V * d == 38_404_096


def test_workspace_query_and_config_checks(lib):
    n = C.c_size_t()
    assert lib.ad_query_workspace(C.byref(_cfg(synth.BASE)), C.byref(n)) == 0
    small = n.value
    assert lib.ad_query_workspace(C.byref(_cfg(synth.BASE, max_batch=32, max_src=64, max_tgt=64, kmax=64)), C.byref(n)) == 0
    assert n.value > small > 0
    bad = _cfg(synth.BASE, kmax=300)
    assert lib.ad_query_workspace(C.byref(bad), C.byref(n)) == binding.AD_ERR_ARG
    assert b"kmax" in lib.ad_last_error(None)
    bad = _cfg(synth.BASE)
    bad.n_heads = 7
    assert lib.ad_query_workspace(C.byref(bad), C.byref(n)) == binding.AD_ERR_ARG
    for d_ffn, rc in ((510, binding.AD_ERR_ARG), (508, binding.AD_OK)):      # vectors are read 16 bytes at a time
        odd = _cfg(synth.TINY)
        odd.d_ffn = d_ffn
        assert lib.ad_query_workspace(C.byref(odd), C.byref(n)) == rc
    bad = _cfg(synth.BASE)
    bad.eos = 40000
    assert lib.ad_query_workspace(C.byref(bad), C.byref(n)) == binding.AD_ERR_ARG


def test_partial_sums_take_no_more_room_than_the_kernels_that_leave_them(lib):
    """FP32 models: the sums per head and per slice of hidden features belong to kernels for passes of up to 1024 tokens and models 128 and
    256 wide; a handle of thousands of tokens, or of another width, has no use for more of them."""
    def size(d, heads, ffn, **kw):
        n = C.c_size_t()
        shape = synth.ModelShape("size", d, heads, ffn, 1000, 1, 1, "fp32")
        assert lib.ad_query_workspace(C.byref(_cfg(shape, **kw)), C.byref(n)) == 0
        return n.value

    slack = 1 << 14                                           # alignment of the buffers
    for d in (128, 256):                                      # twice the heads: so many more sums, with a drafter in both sets of buffers
        for drafter in (0, 1):
            large = dict(max_batch=256, max_src=256, max_tgt=64, kmax=64, has_drafter=drafter)
            more = size(d, d // 32, 1024, **large) - size(d, d // 64, 1024, **large)
            assert 0 < more <= (1 + drafter) * (d // 64) * 1024 * d * 4 + slack
    # 512 wide: none at all, so a slightly wider model needs more room and not less
    some = dict(max_batch=32, max_src=32, max_tgt=32, kmax=32)
    assert size(512, 8, 2048, **some) < size(576, 9, 2048, **some)


def test_struct_layouts():
    assert C.sizeof(binding.ModelCfg) == 17 * 4
    assert C.sizeof(binding.GenOpts) == 40
    assert C.sizeof(binding.Stats) == 48


def test_null_handle_calls_are_rejected(lib):
    assert lib.ad_encode(None, None, 1, None, 1, 1) == binding.AD_ERR_ARG
    assert lib.ad_commit(None, None, 1) == binding.AD_ERR_ARG
    assert lib.ad_destroy(None) == binding.AD_ERR_ARG


@pytest.mark.parametrize("d,heads,ffn,vocab", [(512, 8, 2048, 2048), (512, 8, 2048, 1536), (512, 8, 512, 512), (256, 4, 1024, 1024),
                                               (256, 4, 1024, 768), (1024, 16, 4096, 3072), (768, 12, 3072, 3072), (512, 8, 2048, 32000)])
def test_projection_launches_cover_every_token_count(lib, d, heads, ffn, vocab):
    """Grid and shared memory of every projection of a verification pass against what its launch rule asks for at any token
    count, for vocabularies as large as another projection's output: the two share (N, K) and nothing else."""
    for batch, kmax in ((1, 40), (2, 64), (3, 50), (5, 40), (32, 64), (75, 61)):
        cfg = binding.ModelCfg(d, heads, ffn, vocab, 2, 2, 1, batch, 64, 64, kmax, 0, 1, 2, 3, 1e-5, 0)
        rows, n = (C.c_int32 * (7 * 16))(), C.c_int32()
        assert lib.ad_debug_projection_shapes(C.byref(cfg), rows, 16, C.byref(n)) == 0
        assert n.value >= 1
        for i in range(n.value):
            epi, N, K, ctas, need_ctas, smem, need_smem = rows[7 * i: 7 * i + 7]
            assert ctas >= need_ctas and smem >= need_smem, (batch * kmax, epi, N, K, ctas, need_ctas, smem, need_smem)


@pytest.mark.parametrize("d,vocab,batch,kmax,want", [(512, 16000, 2, 50, 2 * 125), (1024, 18816, 2, 64, 2 * 147), (768, 8192, 2, 33, 2 * 64), (512, 4096, 2, 64, 4 * 32),
                                                     (512, 18944, 2, 64, 148)])
def test_projections_of_65_to_128_tokens_read_their_weights_twice_where_tiles_of_32_tokens_outnumber_the_sms(lib, d, vocab, batch, kmax, want):
    """CTAs of the projection onto vocabularies of fewer feature tiles than there are SMs (148 without a device), and of as many."""
    cfg = binding.ModelCfg(d, d // 64, 2 * d, vocab, 2, 2, 1, batch, 64, 64, kmax, 0, 1, 2, 3, 1e-5, 0)
    rows, n = (C.c_int32 * (7 * 16))(), C.c_int32()
    assert lib.ad_debug_projection_shapes(C.byref(cfg), rows, 16, C.byref(n)) == 0
    ctas = [rows[7 * i + 3] for i in range(n.value) if rows[7 * i] == 3]      # EPI_ARGMAX
    assert ctas == [want]
