"""Contracts of the C ABI that the results alone do not show: workspace sizes that grow with their arguments, inputs
written on the stream just before a call, alignment of caller buffers."""
import pytest
import torch

from paper_2607_20357_gb300 import svl, synth

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

TINY = synth.WORKLOADS["tiny"]
LLAVA = synth.WORKLOADS["llava"]


@pytest.fixture(scope="module")
def deep():
    """LLaVA-7B widths and depth (every layer the same tensors: only sizes and small batches are looked at)."""
    dims = synth.reduced(LLAVA.dims, vocab=512)
    w = synth.make_weights(dims, 1, device="cuda", layers=[0])
    w["layers"] = w["layers"] * dims.n_layers
    m = svl.GatedPrefill(dims, w, max_seq=1024)
    yield m
    m.close()


def test_workspace_sizes_grow_with_every_argument(deep):
    """A workspace sized for a batch serves every smaller one, also across the row count up to which the narrow launches
    of decode run (their QKV list has more tiles a row)."""
    h = deep.handle
    decode = [svl.svl_decode_workspace_size(h, B) for B in range(1, 81)]
    assert decode == sorted(decode)
    for B in (1, 2, 8, 16, 32, 64):
        rows = [svl.svl_workspace_size_for(h, ("prefill",), B, n, 0) for n in range(0, 200)]
        assert rows == sorted(rows), B
        host = [svl.svl_host_workspace_size(h, B, n, 8) for n in range(0, 100)]
        assert host == sorted(host), B
    for n in (0, 1, 16, 24, 31, 32, 33, 64):
        batch = [svl.svl_workspace_size_for(h, ("prefill",), B, n, 0) for B in range(1, 100)]
        assert batch == sorted(batch), n


@pytest.mark.parametrize("sized_for", [33, 36])
def test_decode_of_32_samples_in_a_workspace_of_more(deep, sized_for):
    d, B, max_len = deep.dims, 32, 4
    ws = torch.empty(svl.svl_decode_workspace_size(deep.handle, sized_for), dtype=torch.uint8, device="cuda")
    kv = torch.zeros(svl.svl_kv_cache_size(deep.handle, B, max_len) // 2, dtype=torch.bfloat16, device="cuda")
    i32 = dict(dtype=torch.int32, device="cuda")
    tok, length, nxt = torch.arange(B, **i32), torch.zeros(B, **i32), torch.empty(B, **i32)
    lg = torch.ones(B, d.n_layers, dtype=torch.uint8, device="cuda")
    gg = torch.ones(B, d.n_layers, d.n_groups, dtype=torch.uint8, device="cuda")
    logits = torch.empty(B, d.vocab, device="cuda")
    svl.svl_decode_step(deep.handle, B, tok, kv, max_len, length, lg, gg, logits, nxt, ws, ws.numel())
    assert svl.svl_get_device_status(deep.handle) == 0
    assert length.tolist() == [1] * B and torch.equal(nxt.long(), logits.argmax(1))


# Calls are stream-ordered: what the launch before a call writes is an input like any other, although the library's
# kernels start before their predecessor has ended. A pack whose projector is the identity makes such a predecessor:
# it lets its successor start at once and then writes rows of X, which the next call reads.
def _packer(rows, seed):
    """A model and a batch of one sample whose pack writes `rows` text rows (embedding rows, so any bf16 data) to X."""
    w = synth.make_weights(TINY.dims, seed, device="cuda")
    m = svl.GatedPrefill(TINY.dims, w, max_seq=1024)
    b = synth.make_batch(TINY, seed, n_vis_list=[1], s_text_list=[rows], keep_list=[0], device="cuda")
    out = m.run(b, stages=("select", "pack"))
    torch.cuda.synchronize()
    assert torch.equal(out["X"][:rows], w["embed"][b["text_ids"].long()])
    return m, b, out


def test_quantiser_reads_a_gain_written_by_the_launch_before():
    m, b, out = _packer(16, 91)
    cols = 16 * TINY.dims.d_model  # one gain vector from 16 rows of X
    gain = out["X"][:16].view(-1).clone()
    src = torch.randn(64, cols, device="cuda", generator=torch.Generator("cuda").manual_seed(92)).to(torch.bfloat16)

    def quant(g):
        codes, scale = torch.zeros(64, cols, dtype=torch.uint8, device="cuda"), torch.zeros(64, device="cuda")
        svl.svl_quantize_rows_e4m3(src, 64, cols, cols, codes, cols, scale, gain=g)
        return codes, scale

    want = quant(gain)
    torch.cuda.synchronize()
    for _ in range(20):
        out["X"].zero_()
        torch.cuda.synchronize()
        m.run(b, out=out, stages=("pack",))
        got = quant(out["X"][:16])
        torch.cuda.synchronize()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    m.close()


def test_controller_reads_budget_weights_written_by_the_launch_before():
    packer, b, out = _packer(32, 93)
    dims = synth.reduced(LLAVA.dims, n_layers=1, vocab=512)
    w = synth.make_weights(dims, 94, device="cuda")
    H, X = dims.h_ctrl, out["X"]
    rows = H * H // TINY.dims.d_model  # bud_w1 and bud_w2 are rows of X
    w["bud_w1"], w["bud_w2"] = X[:rows].view(H, H), X[rows:2 * rows].view(H, H)
    m = svl.GatedPrefill(dims, w, max_seq=1024)
    batch = synth.make_batch(LLAVA, 95, batch=4, dims=dims, budget_list=[0.2, 0.5, 0.7, 1.0], device="cuda")
    got = m.run(batch, stages=("select",))
    torch.cuda.synchronize()
    want = {k: got[k].clone() for k in ("scores", "k", "kept_idx", "kept_off")}
    assert float(want["scores"].std()) > 0
    for _ in range(20):
        X.zero_()
        torch.cuda.synchronize()
        packer.run(b, out=out, stages=("pack",))
        m.run(batch, out=got, stages=("select",))
        torch.cuda.synchronize()
        for key in ("scores", "k", "kept_off"):
            assert torch.equal(got[key], want[key]), key
        n = int(want["kept_off"][-1])
        assert torch.equal(got["kept_idx"][:n], want["kept_idx"][:n])
    m.close()
    packer.close()


def test_decode_with_logits_aligned_to_a_float_only():
    """Logits that start 4 bytes past a 16-byte boundary, a vocabulary that is a multiple of four."""
    dims = synth.reduced(TINY.dims, vocab=1024)
    m = svl.GatedPrefill(dims, synth.make_weights(dims, 96, device="cuda"), max_seq=64)
    B, V, max_len = 3, dims.vocab, 8
    i32 = dict(dtype=torch.int32, device="cuda")
    lg = torch.ones(B, dims.n_layers, dtype=torch.uint8, device="cuda")
    gg = torch.ones(B, dims.n_layers, dims.n_groups, dtype=torch.uint8, device="cuda")
    ws = torch.empty(svl.svl_decode_workspace_size(m.handle, B), dtype=torch.uint8, device="cuda")

    def step(logits):
        kv = torch.zeros(svl.svl_kv_cache_size(m.handle, B, max_len) // 2, dtype=torch.bfloat16, device="cuda")
        nxt, length = torch.full((B,), -5, **i32), torch.zeros(B, **i32)
        svl.svl_decode_step(m.handle, B, torch.arange(B, **i32), kv, max_len, length, lg, gg, logits, nxt, ws,
                            ws.numel())
        assert svl.svl_get_device_status(m.handle) == 0
        return nxt

    aligned, base = torch.empty(B, V, device="cuda"), torch.empty(B * V + 4, device="cuda")
    want = step(aligned)
    for shift in (1, 2, 3):
        view = base[shift:shift + B * V].view(B, V)
        assert torch.equal(step(view), want) and torch.equal(view, aligned)
        assert torch.equal(want.long(), view.argmax(1))
    m.close()


def test_e4m3_gemm_refuses_column_scales_it_cannot_read():
    """b_scale is read as 16-byte vectors: other alignments are an argument error and launch nothing."""
    m = svl.GatedPrefill(TINY.dims, synth.make_weights(TINY.dims, 97, device="cuda"), max_seq=64)
    M, N, K = 16, 64, 128
    one = 0x38  # e4m3 code of 1
    A, B = (torch.full((n, K), one, dtype=torch.uint8, device="cuda") for n in (M, N))
    a_scale, b_scale = torch.ones(M + 1, device="cuda"), torch.ones(N + 4, device="cuda")
    C, before = torch.zeros(M, N, device="cuda"), svl.svl_launch_count()
    for shift in (1, 2, 3):
        with pytest.raises(svl.SvlError) as e:
            svl.svl_gemm_e4m3(m.handle, A, a_scale, B, b_scale[shift:], M, N, K, C)
        assert e.value.code == 1 and svl.svl_launch_count() == before
    svl.svl_gemm_e4m3(m.handle, A, a_scale[1:], B, b_scale[4:], M, N, K, C)  # rows: any float
    assert svl.svl_get_device_status(m.handle) == 0 and bool((C == K).all())
    m.close()


def test_packs_chained_through_their_rows():
    """A pack whose visual features are the rows another pack writes just before it."""
    first, b, out = _packer(96, 98)
    want = out["X"][:96].clone()
    m = svl.GatedPrefill(TINY.dims, first.w, max_seq=1024)
    b2 = synth.make_batch(TINY, 99, n_vis_list=[96], s_text_list=[5], keep_list=[96], device="cuda")
    b2["vis"] = out["X"][:96]
    got = m.run(b2, stages=("select", "pack"))
    for _ in range(20):
        out["X"].zero_()
        got["X"].zero_()
        torch.cuda.synchronize()
        first.run(b, out=out, stages=("pack",))
        m.run(b2, out=got, stages=("pack",))
        torch.cuda.synchronize()
        assert torch.equal(got["X"][:96], want)
    m.close()
    first.close()


@pytest.mark.parametrize("gates", ["paper", "later"])
def test_recorded_launch_times_do_not_overlap(gates):
    """Each record covers its own launch: together they take no longer than the call. One sample that keeps all of its
    60,000 tokens makes the compaction far longer than the gaps between launches."""
    n = 60000
    m = svl.GatedPrefill(TINY.dims, synth.make_weights(TINY.dims, 103, device="cuda"), max_seq=64)
    b = synth.make_batch(TINY, 104, n_vis_list=[n], s_text_list=[1], keep_list=[n], device="cuda")
    out = m.alloc_outputs(b)
    ws, wsb = m.workspace(1, n, 1, stages=("select",))
    logits = torch.ones(1, TINY.dims.n_layers, TINY.dims.n_groups, device="cuda")
    lg, gg = (out["layer_gate"], out["group_gate"]) if gates == "paper" else (None, None)

    def call():
        svl.svl_score_select_paper(m.handle, 1, n, b["vis"], b["vis_off"], out["text_len"], b["budget"],
                                   b["keep_count"], logits if gates == "paper" else None, out["scores"], out["k"],
                                   out["kept_idx"], out["kept_off"], out["flags"], lg, gg, None, ws, wsb)

    call()
    for _ in range(5):
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        svl.svl_profile_start(m.handle)
        start.record()
        call()
        end.record()
        svl.svl_profile_stop(m.handle)
        end.synchronize()
        launches = svl.svl_profile_launches(m.handle)
        assert [t for t, _ in launches] == ["budget_embed", "score", "select", "select"]
        assert sum(ms for _, ms in launches) <= start.elapsed_time(end), launches
    m.close()


def test_pack_cuts_off_and_reports_rows_past_its_capacity():
    """text_off that promises more rows than n_text_total: the rows past the capacity are cut off (kept visual rows of
    the second sample among them, which the projector then has no place for), the others are as without the cut, and
    the status word says so. Nothing past the capacity is written."""
    dims = synth.reduced(LLAVA.dims, n_layers=1, vocab=512)
    m = svl.GatedPrefill(dims, synth.make_weights(dims, 105, device="cuda"), max_seq=1024)
    b = synth.make_batch(LLAVA, 106, n_vis_list=[100, 140], s_text_list=[200, 40], keep_list=[100, 140], dims=dims,
                         device="cuda")
    out = m.run(b, stages=("select", "pack"))
    assert svl.svl_get_device_status(m.handle) == 0
    want, D, n_text = out["X"].clone(), dims.d_model, 100  # 240 + 100 rows of 480
    cap = 240 + n_text
    ws = torch.full((svl.svl_workspace_size_for(m.handle, ("pack",), 2, 240, n_text),), 0x7F, dtype=torch.uint8,
                    device="cuda")
    X = torch.full((cap + 64, D), 7.0, dtype=torch.bfloat16, device="cuda")
    svl.svl_pack(m.handle, 2, 240, n_text, b["vis"], b["vis_off"], out["kept_idx"], out["kept_off"], b["text_ids"],
                 b["text_off"], X, out["cu_seqlens"], out["pos"], ws, ws.numel())
    assert svl.svl_get_device_status(m.handle) == svl.SVL_DEV_BAD_INDEX
    assert out["cu_seqlens"].tolist() == [0, 300, cap]
    assert torch.equal(X[:cap], want[:cap]) and bool((X[cap:] == 7).all())
    m.close()
