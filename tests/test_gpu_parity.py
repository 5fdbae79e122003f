"""CUDA path vs the CPU oracle, through the C ABI, on seeded synthetic inputs.

Small cases are compared element by element over the whole output (several
128-token tiles plus a ragged tail).  Full-size workloads, in the launch
configuration bench.py times, are compared on sampled rows the oracle computes
one by one.  Integer outputs (alignment spans) must be bit-exact.
"""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_2608_30963_gb300 as kvx
from paper_2608_30963_gb300 import synth

from harness import compare, make_case, oracle_problem, sample_rows

pytestmark = pytest.mark.gpu

SPECS = synth.config_specs()
PATHS = [kvx.KVX_PATH_SIMT, kvx.KVX_PATH_AUTO]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    kvx.build()
    yield


def _run(c, path, paged=None, max_position=0):
    from gpu_harness import DeviceCase
    g = DeviceCase(c, path=path, paged=paged, max_position=max_position)
    g.run()
    torch.cuda.synchronize()
    return g


def _full_compare(c, path, paged=None, max_position=0):
    g = _run(c, path, paged, max_position)
    ok, ov = oracle_problem(c).translate()
    gk, gv = g.gather()
    sk = compare(gk, ok, c.spec.dtype)
    sv = compare(gv, ov, c.spec.dtype)
    assert g.status() == 0
    return g, sk, sv


def _shrink(spec, Ls, Lt, **kw):
    return dataclasses.replace(spec, src=dataclasses.replace(spec.src, num_layers=Ls),
                               dst=dataclasses.replace(spec.dst, num_layers=Lt), **kw)


# ------------------------------------------------------------------ small, whole output
def test_tiny_fp32_full():
    c = make_case(SPECS["tiny_fp32"])
    _, sk, sv = _full_compare(c, kvx.KVX_PATH_AUTO)
    assert sk["max_abs"] < 1e-4 and sv["max_abs"] < 1e-4


SMALL = {
    # name: (base spec, Ls, Lt, target lengths)
    "qwen7b_qwen1p5b": ("qwen7b_to_qwen1p5b_4k", 3, 3, [300]),
    "qwen1p5b_gemma2b": ("qwen1p5b_to_gemma2b_1k", 4, 3, [300]),
    "llama70b_qwen7b": ("llama70b_to_qwen7b_8k", 9, 4, [300]),
    "longctx_paged_varlen": ("longctx_8k_b4", 2, 2, [37, 300, 129, 1]),
}


@pytest.mark.parametrize("path", PATHS, ids=["simt", "auto"])
@pytest.mark.parametrize("name", list(SMALL))
def test_small_full_output(name, path):
    base, Ls, Lt, lens = SMALL[name]
    spec = _shrink(SPECS[base], Ls, Lt)
    c = make_case(spec, lens, pad_value=float("nan"))
    _full_compare(c, path)


@pytest.mark.parametrize("path", PATHS, ids=["simt", "auto"])
def test_explicit_positions_and_layer_map(path):
    spec = _shrink(SPECS["llama70b_to_qwen7b_8k"], 5, 3, layer_map=[4, 0, 2])
    wl = synth.make_workload(spec, [200, 77])
    rng = np.random.default_rng(3)
    src_pos = rng.integers(0, 120000, size=(wl.batch, wl.s_max)).astype(np.int32)
    tgt_pos = (np.arange(wl.total_tgt) * 7 + 3000).astype(np.int32)
    c = make_case(spec, [200, 77], src_pos=src_pos, tgt_pos=tgt_pos)
    _full_compare(c, path, max_position=1 << 17)


LINEAR4 = dict(rope_type=synth.ROPE_LINEAR, rope_factor=4.0)
SCHEDULES = {
    # Llama-3.1 scaled source RoPE, cross-tokenizer (span kernel)
    "llama3_src_spans": ("llama70b_to_qwen7b_8k", 5, 3, [300, 41], dict(src=synth.LLAMA70B_SCALED), {}),
    # linear target schedule, identity alignment: source and target rotations differ
    "linear_dst_identity": ("qwen7b_to_qwen1p5b_4k", 2, 2, [300, 5], {}, LINEAR4),
    # the same scaled schedule on both sides: source and target rotations coincide
    "llama3_both_identity": ("qwen7b_to_qwen1p5b_4k", 2, 2, [300],
                             dict(rope_type=synth.ROPE_LLAMA3, rope_factor=8.0, rope_low_freq_factor=1.0,
                                  rope_high_freq_factor=4.0, rope_original_max_position=256),
                             dict(rope_type=synth.ROPE_LLAMA3, rope_factor=8.0, rope_low_freq_factor=1.0,
                                  rope_high_freq_factor=4.0, rope_original_max_position=256)),
}


@pytest.mark.parametrize("path", PATHS, ids=["simt", "auto"])
@pytest.mark.parametrize("name", list(SCHEDULES))
def test_rope_schedules(name, path):
    base, Ls, Lt, lens, src_kw, dst_kw = SCHEDULES[name]
    spec = _shrink(SPECS[base], Ls, Lt)
    src = src_kw.get("src", dataclasses.replace(spec.src, **{k: v for k, v in src_kw.items() if k != "src"}))
    src = dataclasses.replace(src, num_layers=Ls)
    spec = dataclasses.replace(spec, src=src, dst=dataclasses.replace(spec.dst, **dst_kw))
    c = make_case(spec, lens, pad_value=float("nan"))
    _full_compare(c, path)


PARTIAL = {
    # (base, Ls, Lt, target lengths, source rotary_dim, target geometry changes); identity
    # alignment with a partial rotary head runs on the span kernel (the identity kernel
    # rotates whole heads only)
    # same partial head on both sides
    "both64_identity": ("qwen7b_to_qwen1p5b_4k", 2, 2, [300, 5], 64, dict(rotary_dim=64)),
    # a quarter of the source head rotates, the target head fully: source side only
    "src32_identity": ("qwen7b_to_qwen1p5b_4k", 2, 2, [300], 32, {}),
    # d_t = 256 in two output tiles, 96 rotating channels: row stores split in up to four runs
    "dst96_identity_split": ("qwen7b_to_qwen1p5b_4k", 2, 2, [300, 41], 0,
                             dict(head_dim=256, rope_base=1e4, rotary_dim=96)),
    # cross-tokenizer spans: partial source (lanes past rhalf do not rotate), partial target
    "src64_spans": ("llama70b_to_qwen7b_8k", 5, 3, [300, 41], 64, {}),
    "dst128_spans_gemma": ("qwen1p5b_to_gemma2b_1k", 3, 2, [300], 0, dict(rotary_dim=128)),
    # fp32 caches: the CUDA-core kernel
    "both32_tiny_fp32": ("tiny_fp32", 4, 2, [256, 100], 32, dict(rotary_dim=32)),
}


@pytest.mark.parametrize("path", PATHS, ids=["simt", "auto"])
@pytest.mark.parametrize("name", list(PARTIAL))
def test_partial_rotary_heads(name, path):
    base, Ls, Lt, lens, rot_s, dst_kw = PARTIAL[name]
    spec = _shrink(SPECS[base], Ls, Lt)
    spec = dataclasses.replace(spec, src=dataclasses.replace(spec.src, rotary_dim=rot_s),
                               dst=dataclasses.replace(spec.dst, **dst_kw))
    c = make_case(spec, lens, pad_value=float("nan"))
    g, _, _ = _full_compare(c, path)
    if path == kvx.KVX_PATH_AUTO and spec.dtype == "bf16":
        assert g.tr.info().path == kvx.KVX_PATH_TCGEN05


FORMS = {
    # one map per target layer over all 8 source heads: in = 1024, streamed weight pieces
    "dense_in1024_spans": ("llama70b_to_qwen7b_8k_dense", 5, 3, [300, 41], {}),
    # dense over 2 source heads (in = 256, resident weights), expansion-shaped geometry, spans
    "dense_in256_spans": ("qwen1p5b_to_gemma2b_1k", 3, 2, [300], dict(form=synth.FORM_DENSE)),
    # dense in = 256 with identity alignment (tensor-TMA kernel)
    "dense_in256_identity": ("qwen7b_to_qwen1p5b_4k", 2, 2, [300, 5],
                             dict(form=synth.FORM_DENSE, src=synth.QWEN1P5B)),
    # groups of two source layers: in = 512, streamed weight pieces
    "layers2_in512_spans": ("llama70b_to_qwen7b_8k_layers2", 5, 3, [300, 41],
                            dict(layer_map=[[0, 1], [2, 3], [4, 4]])),
    # latent adapters, identity alignment and spans
    "latent64_identity": ("qwen7b_to_qwen1p5b_4k_latent64", 2, 2, [300, 5], {}),
    "latent16_spans": ("llama70b_to_qwen7b_8k", 5, 3, [300], dict(rank=16)),
}


@pytest.mark.parametrize("path", PATHS, ids=["simt", "auto"])
@pytest.mark.parametrize("name", list(FORMS))
def test_translator_forms(name, path):
    base, Ls, Lt, lens, kw = FORMS[name]
    spec = _shrink(SPECS[base], Ls, Lt)
    kw = dict(kw)
    if "src" in kw:
        kw["src"] = dataclasses.replace(kw["src"], num_layers=Ls)
    spec = dataclasses.replace(spec, **kw)
    c = make_case(spec, lens, pad_value=float("nan"))
    g, _, _ = _full_compare(c, path)
    if path == kvx.KVX_PATH_AUTO:
        assert g.tr.info().path == kvx.KVX_PATH_TCGEN05


HEAD_DIMS = {
    # source / target head dims other than 128: every instantiation of the tensor-core kernels
    "ds64_dt64": (synth.ModelGeom(2, 4, 64, 1e4), synth.ModelGeom(2, 2, 64, 1e4)),
    "ds256_dt128": (synth.ModelGeom(2, 2, 256, 1e4), synth.ModelGeom(2, 2, 128, 1e6)),
    "ds256_dt256_expand": (synth.ModelGeom(2, 1, 256, 1e6), synth.ModelGeom(2, 2, 256, 1e4)),
    "ds64_dt256": (synth.ModelGeom(3, 4, 64, 1e6), synth.ModelGeom(2, 1, 256, 1e4)),
}


@pytest.mark.parametrize("path", PATHS, ids=["simt", "auto"])
@pytest.mark.parametrize("spans", [False, True], ids=["identity", "spans"])
@pytest.mark.parametrize("name", list(HEAD_DIMS))
def test_head_dims(name, spans, path):
    src, dst = HEAD_DIMS[name]
    spec = synth.WorkloadSpec(name, src, dst, "bf16", [300], spans, None, True)
    c = make_case(spec, [300, 77], pad_value=float("nan"))
    g, _, _ = _full_compare(c, path)
    if path == kvx.KVX_PATH_AUTO:
        assert g.tr.info().path == kvx.KVX_PATH_TCGEN05


def test_tiny_token_counts_and_empty_sequences():
    spec = _shrink(SPECS["qwen1p5b_to_gemma2b_1k"], 2, 2)
    c = make_case(spec, [1, 0, 2, 0, 129])
    for path in PATHS:
        _full_compare(c, path)


# ------------------------------------------------------------------ invariances (bit-exact)
@pytest.mark.parametrize("path", PATHS, ids=["simt", "auto"])
def test_paged_equals_contiguous_and_batch_invariance(path):
    spec = _shrink(SPECS["longctx_8k_b4"], 2, 2)
    c = make_case(spec, [37, 300, 129])
    gp = _run(c, path, paged=True)
    gc = _run(c, path, paged=False)
    pk, pv = gp.gather()
    ck, cv = gc.gather()
    np.testing.assert_array_equal(pk, ck)
    np.testing.assert_array_equal(pv, cv)
    solo = make_case(spec, [300])
    # the second sequence alone: same source rows, same weights
    for l in solo.src_k:
        solo.src_k[l] = c.src_k[l][1:2, :, :300]
        solo.src_v[l] = c.src_v[l][1:2, :, :300]
    gs = _run(solo, path, paged=False)
    sk, sv = gs.gather()
    np.testing.assert_array_equal(sk, ck[:, :, 37:337])
    np.testing.assert_array_equal(sv, cv[:, :, 37:337])


# ------------------------------------------------------------------ full-size, sampled rows
FULL = ["qwen7b_to_qwen1p5b_4k", "qwen1p5b_to_gemma2b_1k", "qwen1p5b_to_gemma2b_2k", "qwen1p5b_to_gemma2b_4k",
        "llama70b_to_qwen7b_8k", "longctx_8k_b4", "tiny_fp32", "llama70b_to_qwen7b_8k_dense",
        "qwen7b_to_qwen1p5b_4k_latent64"]


def test_layer_groups_8k_sampled():
    """Groups of two source layers at the full 8K context, on 6 target layers (the full
    28-layer map would hold 56 source layers in host memory)."""
    spec = dataclasses.replace(SPECS["llama70b_to_qwen7b_8k_layers2"],
                               dst=dataclasses.replace(SPECS["llama70b_to_qwen7b_8k_layers2"].dst, num_layers=6),
                               layer_map=synth.layer_groups(80, 6, 2))
    c = make_case(spec)
    g = _run(c, kvx.KVX_PATH_AUTO)
    p = oracle_problem(c)
    rows = sample_rows(c, 300)
    compare(np.stack([g.row(*r) for r in rows]), np.stack([p.row(*r) for r in rows]), "bf16")
    assert g.status() == 0


@pytest.mark.parametrize("name", FULL)
def test_full_size_sampled(name):
    c = make_case(SPECS[name])
    g = _run(c, kvx.KVX_PATH_AUTO)
    p = oracle_problem(c)
    rows = sample_rows(c, 400)
    gpu = np.stack([g.row(*r) for r in rows])
    ref = np.stack([p.row(*r) for r in rows])
    compare(gpu, ref, c.spec.dtype)
    assert g.status() == 0


# ------------------------------------------------------------------ alignment builder
@pytest.mark.parametrize("key,ms,mt", [(0, 4.0, 4.0), (1, 5.0, 2.0), (2, 2.0, 6.0), (3, 1.0, 1.0)])
def test_alignment_builder_bit_exact(key, ms, mt):
    from gpu_harness import i32
    src_ends, tgt_ends = [], []
    for i, nb in enumerate([1, 57, 5000, 911]):
        se, te = synth.draw_tokenizations(nb, ms, mt, key * 10 + i)
        src_ends.append(se); tgt_ends.append(te)
    so = np.concatenate([[0], np.cumsum([len(x) for x in src_ends])]).astype(np.int32)
    to = np.concatenate([[0], np.cumsum([len(x) for x in tgt_ends])]).astype(np.int32)
    se, te = np.concatenate(src_ends), np.concatenate(tgt_ends)
    lo_ref, hi_ref, n = oracle.build_alignment(so, se, to, te)
    T = int(to[-1])
    lo = torch.full((T,), -7, dtype=torch.int32, device="cuda")
    hi = torch.full((T,), -7, dtype=torch.int32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    kvx.build_alignment(i32(so), i32(se), i32(to), i32(te), lo, hi, st)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(lo.cpu().numpy(), lo_ref)
    np.testing.assert_array_equal(hi.cpu().numpy(), hi_ref)
    assert int(st.item()) == 0 and n == 0


def test_alignment_builder_recovers_generated_spans():
    from gpu_harness import i32
    spec = SPECS["qwen1p5b_to_gemma2b_4k"]
    wl = synth.make_workload(spec, [4096, 1000, 3])
    T = wl.total_tgt
    lo = torch.empty(T, dtype=torch.int32, device="cuda")
    hi = torch.empty(T, dtype=torch.int32, device="cuda")
    kvx.build_alignment(i32(wl.src_seq_off), i32(wl.src_end), i32(wl.tgt_seq_off), i32(wl.tgt_end), lo, hi)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(lo.cpu().numpy(), wl.span_lo)
    np.testing.assert_array_equal(hi.cpu().numpy(), wl.span_hi)


# ------------------------------------------------------------------ device status (no faults)
@pytest.mark.parametrize("path", PATHS, ids=["simt", "auto"])
def test_bad_spans_pages_positions_set_status_bits(path):
    from gpu_harness import DeviceCase, i32
    spec = _shrink(SPECS["longctx_8k_b4"], 2, 2)
    c = make_case(spec, [40, 20])
    g = DeviceCase(c, path=path, paged=True)
    T = c.wl.total_tgt
    lo = np.arange(T, dtype=np.int32) - np.repeat(c.wl.tgt_seq_off[:-1], c.wl.tgt_len)
    hi = lo + 1
    hi[5] = 10_000          # past the source length
    g.span_lo, g.span_hi = i32(lo), i32(hi)
    g.run()
    assert g.status() & kvx.KVX_DEV_SPAN_CLAMPED
    g.span_lo = g.span_hi = None
    pt = c.wl.page_table.copy()
    pt[1, 0] = 10_000       # page outside the pool
    g.page_table = i32(pt)
    g.run()
    assert g.status() == kvx.KVX_DEV_PAGE_INVALID
    g.page_table = i32(c.wl.page_table)
    g.tgt_pos = i32(np.full(T, 1 << 30, np.int32))
    g.run()
    assert g.status() == kvx.KVX_DEV_POS_CLAMPED
    g.tgt_pos = None
    g.run()
    assert g.status() == 0


def test_invalid_arguments_rejected_before_launch():
    from gpu_harness import DeviceCase
    spec = _shrink(SPECS["qwen7b_to_qwen1p5b_4k"], 2, 2)
    c = make_case(spec, [64])
    g = DeviceCase(c)
    g.span_hi = None          # span_lo without span_hi
    g.span_lo = g.seq_off
    with pytest.raises(kvx.KvxError) as e:
        g.run()
    assert e.value.status == kvx.KVX_ERR_INVALID_ARG
    bad = synth.ModelGeom(2, 3, 128, 1e6)
    with pytest.raises(kvx.KvxError) as e:
        kvx.Translator(bad, spec.dst, torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda"))
    assert e.value.status == kvx.KVX_ERR_UNSUPPORTED


# ------------------------------------------------------------------ the two tensor-core kernels agree
@pytest.mark.parametrize("base,Ls,Lt,lens", [("qwen7b_to_qwen1p5b_4k", 2, 2, [300, 5, 129]),
                                             ("qwen1p5b_to_gemma2b_1k", 2, 2, [300]),
                                             ("llama70b_to_qwen7b_8k", 3, 2, [257])])
def test_identity_kernel_equals_span_kernel(base, Ls, Lt, lens):
    """Identity alignment (no span arrays) runs the tensor-TMA kernel; the same
    spans given explicitly run the span-gather kernel.  Same arithmetic: equal bits."""
    from gpu_harness import i32
    spec = _shrink(SPECS[base], Ls, Lt, cross_tokenizer=False)
    c = make_case(spec, lens)
    ga = _run(c, kvx.KVX_PATH_AUTO)
    from gpu_harness import DeviceCase
    gs = DeviceCase(c, path=kvx.KVX_PATH_AUTO)
    lo = np.concatenate([np.arange(t, dtype=np.int32) for t in lens])
    gs.span_lo, gs.span_hi = i32(lo), i32(lo + 1)
    gs.run()
    torch.cuda.synchronize()
    ak, av = ga.gather()
    sk, sv = gs.gather()
    np.testing.assert_array_equal(ak, sk)
    np.testing.assert_array_equal(av, sv)
    assert ga.status() == 0 and gs.status() == 0


# ------------------------------------------------------------------ largest workload: properties + sampled rows
def test_longctx_32k_b8_device_generated():
    """The 32K x 8 paged workload (~196K target tokens).  Inputs are drawn on the device
    from a fixed seed (host fp32 copies would need ~30 GB).  Checks, bit-exact: paged ==
    contiguous and identity kernel == span kernel (explicit identity spans); and sampled
    rows against the oracle, which reads the sampled layers copied back to the host."""
    from gpu_harness import i32, to_host
    spec = SPECS["longctx_32k_b8"]
    wl = synth.make_workload(spec)
    s, d = spec.src, spec.dst
    gen = torch.Generator(device="cuda").manual_seed(20260)
    shape = (wl.batch, s.num_kv_heads, wl.s_max, s.head_dim)
    ks = [torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16) for _ in range(s.num_layers)]
    vs = [torch.randn(shape, generator=gen, device="cuda").to(torch.bfloat16) for _ in range(s.num_layers)]
    w_k = torch.randn((d.num_layers, d.num_kv_heads, spec.group_in, d.head_dim), generator=gen, device="cuda")
    w_v = torch.randn((d.num_layers, d.num_kv_heads, spec.group_in, d.head_dim), generator=gen, device="cuda")
    w_k = (w_k / spec.group_in ** 0.5).to(torch.bfloat16)
    w_v = (w_v / spec.group_in ** 0.5).to(torch.bfloat16)
    lm = list(range(d.num_layers))
    tr = kvx.Translator(s, d, w_k, w_v, layer_map=lm)
    src_len, seq_off = i32(wl.src_len), i32(wl.tgt_seq_off)
    T = wl.total_tgt
    pt = i32(wl.page_table)
    pool = (wl.num_pages, spec.page_size, d.num_kv_heads, d.head_dim)
    cont = (wl.batch, d.num_kv_heads, wl.t_max, d.head_dim)
    pk = [torch.full(pool, float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(d.num_layers)]
    pv = [torch.full(pool, float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(d.num_layers)]
    tr.translate(ks, vs, src_len, seq_off, T, pk, pv, page_table=pt, page_size=spec.page_size,
                 num_pages=wl.num_pages)
    assert tr.device_status() == 0
    ck = [torch.full(cont, float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(d.num_layers)]
    cv = [torch.full(cont, float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(d.num_layers)]
    tr.translate(ks, vs, src_len, seq_off, T, ck, cv)
    assert tr.device_status() == 0
    lo = np.concatenate([np.arange(t, dtype=np.int32) for t in wl.tgt_len])
    sk_ = [torch.full(cont, float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(3)]
    sv_ = [torch.full(cont, float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(3)]
    # span kernel on three layers (a 3-layer translator over the same source layers 0, 13, 27)
    sub = [0, 13, 27]
    tr3 = kvx.Translator(s, dataclasses.replace(d, num_layers=3), w_k[sub].contiguous(), w_v[sub].contiguous(),
                         layer_map=sub)
    tr3.translate(ks, vs, src_len, seq_off, T, sk_, sv_, span_lo=i32(lo), span_hi=i32(lo + 1))
    assert tr3.device_status() == 0
    torch.cuda.synchronize()
    for b in range(wl.batch):
        n = int(wl.tgt_len[b])
        pages = torch.from_numpy(wl.page_table[b]).cuda().long()
        for j in range(d.num_layers):
            for P_, C_ in ((pk[j], ck[j]), (pv[j], cv[j])):
                idx = torch.arange(n, device="cuda")
                rows = P_[pages[idx // spec.page_size], idx % spec.page_size]       # [n, Ht, dt]
                assert torch.equal(rows.transpose(0, 1).view(torch.int16), C_[b, :, :n].view(torch.int16))
        for i, j in enumerate(sub):
            assert torch.equal(sk_[i][b, :, :n].view(torch.int16), ck[j][b, :, :n].view(torch.int16))
            assert torch.equal(sv_[i][b, :, :n].view(torch.int16), cv[j][b, :, :n].view(torch.int16))
    # sampled rows against the oracle on the three layers
    src_k = {l: to_host(ks[l]) for l in sub}
    src_v = {l: to_host(vs[l]) for l in sub}
    dummy = src_k[0]
    p = oracle.OracleProblem(s, dataclasses.replace(d, num_layers=3), [0, 13, 27], wl.src_len, wl.tgt_seq_off,
                             wl.s_max, wl.t_max, [src_k.get(l, dummy) for l in range(s.num_layers)],
                             [src_v.get(l, dummy) for l in range(s.num_layers)],
                             to_host(w_k[sub]), to_host(w_v[sub]))
    r = np.random.default_rng(5)
    gpu, ref = [], []
    for _ in range(300):
        i, h, kv = int(r.integers(3)), int(r.integers(d.num_kv_heads)), int(r.integers(2))
        tp = int(r.integers(T))
        b = int(np.searchsorted(wl.tgt_seq_off, tp, side="right") - 1)
        t = tp - int(wl.tgt_seq_off[b])
        gpu.append(to_host((ck if kv == 0 else cv)[sub[i]][b, h, t]))
        ref.append(p.row(i, h, kv, tp))
    compare(np.stack(gpu), np.stack(ref), "bf16")


# ------------------------------------------------------------------ graphs and streams
@pytest.mark.parametrize("base,lens", [("qwen7b_to_qwen1p5b_4k", [300, 129]), ("qwen1p5b_to_gemma2b_1k", [300])])
def test_translate_captured_in_a_cuda_graph_equals_eager(base, lens):
    """kvx_translate allocates nothing and never synchronises: captured in a CUDA graph and
    replayed twice, it writes the same bits as an eager call."""
    spec = _shrink(SPECS[base], 2, 2)
    c = make_case(spec, lens)
    g = _run(c, kvx.KVX_PATH_AUTO)
    ek, ev = g.gather()
    for t in g.dst_k + g.dst_v:
        t.fill_(float("nan"))
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        g.run(stream=s)          # warm-up on the capture stream
        s.synchronize()
        for t in g.dst_k + g.dst_v:
            t.fill_(float("nan"))
        with torch.cuda.graph(graph, stream=s):
            g.run(stream=s)
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        gk, gv = g.gather()
        np.testing.assert_array_equal(gk, ek)
        np.testing.assert_array_equal(gv, ev)
    assert g.status() == 0


def test_two_translators_on_two_streams():
    """Two translations in flight at once on two streams write exactly their eager results."""
    a = make_case(_shrink(SPECS["qwen7b_to_qwen1p5b_4k"], 2, 2), [640])
    b = make_case(_shrink(SPECS["llama70b_to_qwen7b_8k"], 5, 3), [500])
    ga, gb = _run(a, kvx.KVX_PATH_AUTO), _run(b, kvx.KVX_PATH_AUTO)
    ref = (ga.gather(), gb.gather())
    for g in (ga, gb):
        for t in g.dst_k + g.dst_v:
            t.fill_(float("nan"))
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    s1.wait_stream(torch.cuda.current_stream())
    s2.wait_stream(torch.cuda.current_stream())
    for _ in range(3):
        ga.run(stream=s1)
        gb.run(stream=s2)
    torch.cuda.synchronize()
    for g, (rk, rv) in zip((ga, gb), ref):
        gk, gv = g.gather()
        np.testing.assert_array_equal(gk, rk)
        np.testing.assert_array_equal(gv, rv)
        assert g.status() == 0


# ------------------------------------------------------------------ limits of the fast paths
@pytest.mark.parametrize("batch", [300, 600])
def test_large_batches(batch):
    """More sequences than the identity kernel keeps on chip (256), and than the span kernel
    caches in shared memory (512): both fall back to their general paths, same results."""
    rng = np.random.default_rng(batch)
    lens = [int(x) for x in rng.integers(1, 24, size=batch)]
    for base in ("qwen7b_to_qwen1p5b_4k", "qwen1p5b_to_gemma2b_1k"):
        spec = _shrink(SPECS[base], 2, 2)
        c = make_case(spec, lens)
        g, _, _ = _full_compare(c, kvx.KVX_PATH_AUTO)
        assert g.tr.info().path == kvx.KVX_PATH_TCGEN05


def test_more_target_layers_than_the_identity_kernel_takes():
    """100 target layers (above the identity kernel's 96): the span kernel serves identity
    alignment too."""
    spec = synth.WorkloadSpec("deep", synth.ModelGeom(120, 2, 64, 1e4), synth.ModelGeom(100, 1, 64, 1e6), "bf16",
                              [40], False, None, False)
    c = make_case(spec, [40, 17])
    _full_compare(c, kvx.KVX_PATH_AUTO)


@pytest.mark.parametrize("dtype", [kvx.KVX_FP32, kvx.KVX_BF16])
@pytest.mark.parametrize("Hs,ds,Ht,dt", [(2, 64, 1, 64), (2, 128, 2, 128), (1, 64, 2, 256)])
def test_cuda_core_tile_sizes_agree(Hs, ds, Ht, dt, dtype):
    """A 40-layer translation of 200 tokens takes 32-token tiles, its first two layers alone 16-token
    tiles (compared with the oracle elsewhere): every output is one accumulator over the inputs in the
    same order, so the two agree bit for bit.  Spans of 1..3 rows, a ragged last tile in both."""
    L, T = 40, 200
    rng = np.random.default_rng(5)
    hi = np.cumsum(rng.choice([1, 2, 3], size=T))
    lo = np.concatenate([[0], hi[:-1]])
    S = int(hi[-1])
    tdt = torch.float32 if dtype == kvx.KVX_FP32 else torch.bfloat16
    i32 = lambda x: torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda *sh: torch.randn(sh, device="cuda", generator=gen).to(tdt)
    n_in = max(1, Hs // Ht) * ds
    src = [[rnd(1, Hs, S, ds) for _ in range(L)] for _ in range(2)]
    w = [rnd(L, Ht, n_in, dt) for _ in range(2)]
    outs = []
    for n in (L, 2):
        tr = kvx.Translator(synth.ModelGeom(L, Hs, ds, 1e4), synth.ModelGeom(n, Ht, dt, 1e6), w[0][:n], w[1][:n],
                            layer_map=list(range(n)), dtype=dtype, path=kvx.KVX_PATH_SIMT)
        dst = [[torch.full((1, Ht, T, dt), float("nan"), dtype=tdt, device="cuda") for _ in range(n)] for _ in range(2)]
        tr.translate(src[0], src[1], i32([S]), i32([0, T]), T, dst[0], dst[1], span_lo=i32(lo), span_hi=i32(hi))
        torch.cuda.synchronize()
        outs.append(dst)
    for kv in range(2):
        for j in range(2):
            assert not outs[0][kv][j].isnan().any()
            assert torch.equal(outs[0][kv][j], outs[1][kv][j]), (kv, j)


@pytest.mark.parametrize("T", [1, 128, 259])
@pytest.mark.parametrize("law", ["one", "two", "nine", "mixed"])
@pytest.mark.parametrize("Hs,ds,Ht,dt", [(1, 64, 1, 64), (4, 64, 1, 128), (2, 128, 1, 64), (1, 128, 2, 256), (1, 256, 1, 128),
                                         (4, 128, 1, 128), (4, 256, 1, 256)])
def test_gathered_rows_kernel_edges(Hs, ds, Ht, dt, law, T):
    """The row-gather kernel against the CUDA-core kernel (itself held to the oracle above): one to four
    source heads of every width (inputs of up to 256 channels, and two and four groups of 256), one token, whole and ragged tiles, two sequences of which the second has
    no source tokens left of its spans, spans of one row, of two, of nine (more further rows than the side
    buffer holds) and of 1..12 overlapping and descending, explicit source positions.  Both sum in fp32;
    the row-gather kernel rounds its input rows to bf16 first, a relative 2^-9 each."""
    rng = np.random.default_rng(17)
    n = {"one": np.ones(T, int), "two": np.full(T, 2), "nine": np.full(T, 9), "mixed": rng.integers(1, 13, size=T)}[law]
    S = 400
    lo = rng.integers(0, S - 12, size=T) if law == "mixed" else np.minimum(np.cumsum(n) - n, S - 9)
    i32 = lambda x: torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(3)
    rnd = lambda *sh: torch.randn(sh, device="cuda", generator=gen).to(torch.bfloat16)
    L, n_in = 3, max(1, Hs // Ht) * ds
    src = [[rnd(2, Hs, S, ds) for _ in range(L)] for _ in range(2)]
    w = [rnd(L, Ht, n_in, dt) for _ in range(2)]
    t0 = T - T // 3                      # the second sequence's tokens: its source is empty
    pos = i32(rng.permutation(2 * S))
    outs = []
    for path in (kvx.KVX_PATH_AUTO, kvx.KVX_PATH_SIMT):
        tr = kvx.Translator(synth.ModelGeom(L, Hs, ds, 1e4), synth.ModelGeom(L, Ht, dt, 1e6), w[0], w[1],
                            layer_map=list(range(L)), path=path)
        dst = [[torch.full((2, Ht, T, dt), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(L)] for _ in range(2)]
        tr.translate(src[0], src[1], i32([S, 0]), i32([0, t0, T]), T, dst[0], dst[1], span_lo=i32(lo), span_hi=i32(lo + n),
                     src_pos=pos)
        torch.cuda.synchronize()
        outs.append(torch.stack([torch.stack(d) for d in dst]).double())
    a, b = outs
    assert torch.equal(a.isnan(), b.isnan())          # the same rows written
    a, b = a.nan_to_num(), b.nan_to_num()
    assert a[:, :, 1].abs().max() == 0 and b[:, :, 1].abs().max() == 0   # no source tokens: zero rows
    for kv in range(2):
        assert (a[kv] - b[kv]).norm() <= 2.0 ** -8 * 1.5 * b[kv].norm(), (kv, (a[kv] - b[kv]).norm() / b[kv].norm())


@pytest.mark.parametrize("spans", [False, True])
@pytest.mark.parametrize("Hs,ds,Ht,dt,kl", [(8, 64, 1, 64, 1), (4, 128, 1, 64, 1), (2, 256, 1, 64, 1), (4, 128, 2, 64, 2),
                                            (1, 128, 1, 64, 4), (8, 128, 2, 64, 2), (8, 128, 1, 64, 1), (4, 128, 1, 256, 1)])
def test_inputs_of_several_k_groups_reach_every_channel(Hs, ds, Ht, dt, kl, spans):
    """Inputs of 512 and 1024 channels (one, two and four source layers), with spans and one tokenizer.  512
    onto 64-channel heads has a weight image that would fit shared memory whole, and still takes two K groups.
    Against the CUDA-core kernel: both sum in fp32, the tensor-core kernels round their input rows to bf16
    first, a relative 2^-9 each."""
    L, T = 3, 300
    rng = np.random.default_rng(23)
    n = rng.integers(1, 4, size=T) if spans else np.ones(T, int)
    hi = np.cumsum(n)
    S = int(hi[-1])
    i32 = lambda x: torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(4)
    rnd = lambda *sh: torch.randn(sh, device="cuda", generator=gen).to(torch.bfloat16)
    n_in = kl * max(1, Hs // Ht) * ds
    src = [[rnd(1, Hs, S, ds) for _ in range(L * kl)] for _ in range(2)]
    w = [rnd(L, Ht, n_in, dt) for _ in range(2)]
    sp = dict(span_lo=i32(hi - n), span_hi=i32(hi)) if spans else {}
    outs = []
    for path in (kvx.KVX_PATH_TCGEN05, kvx.KVX_PATH_SIMT):
        tr = kvx.Translator(synth.ModelGeom(L * kl, Hs, ds, 1e4), synth.ModelGeom(L, Ht, dt, 1e6), w[0], w[1],
                            layer_map=[[j * kl + k for k in range(kl)] for j in range(L)], path=path, layers_per_target=kl)
        dst = [[torch.full((1, Ht, T, dt), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(L)] for _ in range(2)]
        tr.translate(src[0], src[1], i32([S]), i32([0, T]), T, dst[0], dst[1], **sp)
        torch.cuda.synchronize()
        assert tr.device_status() == 0
        outs.append(torch.stack([torch.stack(d) for d in dst]).double())
    a, b = outs
    assert not a.isnan().any() and not b.isnan().any()
    for kv in range(2):
        assert (a[kv] - b[kv]).norm() <= 2.0 ** -8 * 1.5 * b[kv].norm(), (kv, (a[kv] - b[kv]).norm() / b[kv].norm())


@pytest.mark.parametrize("Hs,ds,Ht,dt", [(1, 64, 1, 64), (4, 64, 1, 128), (1, 128, 2, 256), (2, 128, 1, 128), (1, 256, 1, 128),
                                         (4, 128, 1, 128)])
@pytest.mark.parametrize("law", ["few_long", "few_long_padded", "all_long", "overlapping", "overlapping_padded"])
def test_span_kernels_agree_on_either_side_of_the_dense_rule(Hs, ds, Ht, dt, law):
    """The row-gather kernel takes calls whose spans mostly fit its side buffer, and runs the window kernel's body on
    dense ones where the source caches may hold 1.5 rows a token.  few_long: 20 spans of 12 rows among 2051 (its own
    walk, whose overflowing tile reads further rows from memory); all_long: 12 rows each; overlapping: three rows
    each, two of them the next token's; padded: caches of twice the length.  Against the CUDA-core kernel, as above."""
    T, L = 2051, 2
    law, padded = law.removesuffix("_padded"), law.endswith("_padded")
    n = np.full(T, {"few_long": 1, "all_long": 12, "overlapping": 3}[law])
    if law == "few_long":
        n[700:720] = 12
    lo = np.arange(T) if law == "overlapping" else np.cumsum(n) - n
    S = int((lo + n).max())
    i32 = lambda x: torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(6)
    rnd = lambda *sh: torch.randn(sh, device="cuda", generator=gen).to(torch.bfloat16)
    n_in = max(1, Hs // Ht) * ds
    src = [[rnd(1, Hs, S * (2 if padded else 1), ds) for _ in range(L)] for _ in range(2)]
    w = [rnd(L, Ht, n_in, dt) for _ in range(2)]
    outs = []
    for path in (kvx.KVX_PATH_TCGEN05, kvx.KVX_PATH_SIMT):
        tr = kvx.Translator(synth.ModelGeom(L, Hs, ds, 1e4), synth.ModelGeom(L, Ht, dt, 1e6), w[0], w[1],
                            layer_map=list(range(L)), path=path)
        dst = [[torch.full((1, Ht, T, dt), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(L)] for _ in range(2)]
        for _ in range(2):   # twice: the second call follows the first on the stream
            tr.translate(src[0], src[1], i32([S]), i32([0, T]), T, dst[0], dst[1], span_lo=i32(lo), span_hi=i32(lo + n))
        torch.cuda.synchronize()
        assert tr.device_status() == 0
        outs.append(torch.stack([torch.stack(d) for d in dst]).double())
    a, b = outs
    assert not a.isnan().any() and not b.isnan().any()
    for kv in range(2):
        assert (a[kv] - b[kv]).norm() <= 2.0 ** -8 * 1.5 * b[kv].norm(), (kv, (a[kv] - b[kv]).norm() / b[kv].norm())


@pytest.mark.parametrize("kw,path,threads", [
    (dict(path=kvx.KVX_PATH_SIMT), kvx.KVX_PATH_SIMT, 128),
    (dict(), kvx.KVX_PATH_TCGEN05, 640),                                       # row gather: 20 warps
    (dict(form=kvx.KVX_FORM_DENSE), kvx.KVX_PATH_TCGEN05, 608),                # windows, weights streamed: 19 warps
    (dict(rotary_dim=64), kvx.KVX_PATH_TCGEN05, 576),                          # windows, weights resident: 18 warps
], ids=["simt", "rows", "windows_streamed", "windows_resident"])
def test_info_reports_the_kernel_that_runs(kw, path, threads):
    kw = dict(kw)
    rd = kw.pop("rotary_dim", 0)
    n_in = 4 * 128 if "form" in kw else 2 * 128
    w = torch.zeros((2, 2, n_in, 128), dtype=torch.bfloat16, device="cuda")
    tr = kvx.Translator(synth.ModelGeom(2, 4, 128, 1e4, rotary_dim=rd), synth.ModelGeom(2, 2, 128, 1e4, rotary_dim=rd), w, w,
                        layer_map=[0, 1], **kw)
    info = tr.info()
    assert (info.path, info.threads, info.num_sms) == (path, threads, torch.cuda.get_device_properties(0).multi_processor_count)
    # 32 tokens of 256 + 4 floats and two blocks of 8 rows of W by 128 channels
    assert info.smem_bytes == (32 * (n_in + 4) * 4 + 2 * 8 * 128 * 4 if path == kvx.KVX_PATH_SIMT else 227 * 1024)


@pytest.mark.parametrize("Hs,ds,Ht,dt", [(4, 64, 2, 256), (4, 64, 4, 256), (2, 64, 2, 256), (2, 128, 2, 128), (2, 64, 4, 128)])
def test_dense_form_with_one_tokenizer(Hs, ds, Ht, dt):
    """The dense form without span arrays: weight images that the identity kernel keeps resident, and 256 channels onto
    256, which it cannot (128 KB).  Against the CUDA-core kernel, as above."""
    L, T = 2, 300
    i32 = lambda x: torch.tensor(np.asarray(x), dtype=torch.int32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(12)
    rnd = lambda *sh: torch.randn(sh, device="cuda", generator=gen).to(torch.bfloat16)
    src = [[rnd(1, Hs, T, ds) for _ in range(L)] for _ in range(2)]
    w = [rnd(L, Ht, Hs * ds, dt) for _ in range(2)]
    outs = []
    for path in (kvx.KVX_PATH_TCGEN05, kvx.KVX_PATH_SIMT):
        tr = kvx.Translator(synth.ModelGeom(L, Hs, ds, 1e4), synth.ModelGeom(L, Ht, dt, 1e6), w[0], w[1],
                            layer_map=list(range(L)), path=path, form=kvx.KVX_FORM_DENSE)
        dst = [[torch.full((1, Ht, T, dt), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(L)] for _ in range(2)]
        tr.translate(src[0], src[1], i32([T]), i32([0, T]), T, dst[0], dst[1])
        torch.cuda.synchronize()
        assert tr.device_status() == 0
        outs.append(torch.stack([torch.stack(d) for d in dst]).double())
    a, b = outs
    assert not a.isnan().any() and not b.isnan().any()
    for kv in range(2):
        assert (a[kv] - b[kv]).norm() <= 2.0 ** -8 * 1.5 * b[kv].norm(), (kv, (a[kv] - b[kv]).norm() / b[kv].norm())
