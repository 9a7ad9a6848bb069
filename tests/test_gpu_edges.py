"""Edges of the kernels' sizes: selection chunks and ties, work lists of many
samples, K-split tails of the residual GEMMs, attention item order, decode
attention with shared KV heads, projector tile shapes, CTA pairs against single
CTAs. Each is compared with plain torch in float64 on the GPU's own inputs, with
the oracle, or with the same work cut differently."""
import numpy as np
import pytest
import torch

from oracle import smartvl_oracle as O
from paper_2607_20357_gb300 import svl, synth
from tests.gpu_common import bar_for, check_selection, rel_err
from tests.test_gpu_decode import _decode
from tests.test_gpu_stages import ACC, check_close, np64

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

TINY = synth.WORKLOADS["tiny"]
LLAVA = synth.WORKLOADS["llava"]
F64 = torch.float64


def _model(dims, seed, **kw):
    w = synth.make_weights(dims, seed, device="cuda")
    return svl.GatedPrefill(dims, w, **kw), w


@pytest.mark.parametrize("lengths", [[1, 31, 512, 0, 513], [4096, 4097], [6000], [40] * 300])
def test_selection_is_the_exact_top_k_of_its_logits(lengths):
    """Keys in shared memory up to 4,096 per sample and in global memory beyond; chunks of 512; many equal logits
    (features repeat), so that ties decide; kept offsets over 300 samples."""
    m, _ = _model(TINY.dims, 5, max_seq=8192)
    b = synth.make_batch(TINY, 6, n_vis_list=[max(n, 1) for n in lengths], s_text_list=[4] * len(lengths),
                         keep_list=[n // 3 for n in lengths], device="cuda")
    off = np.concatenate([[0], np.cumsum(lengths)])
    proto = torch.randn(37, TINY.dims.c_vis, device="cuda", generator=torch.Generator("cuda").manual_seed(7))
    b["vis"] = proto[torch.arange(int(off[-1]), device="cuda") * 7 % 37].to(torch.bfloat16)
    b["vis_off"] = torch.tensor(off, dtype=torch.int32).cuda()
    out = m.run(b, stages=("select",))
    k, ko = out["k"].tolist(), out["kept_off"].tolist()
    assert k == [n // 3 for n in lengths] and ko == [0] + np.cumsum(k).tolist()
    z = out["scores"].double()
    for i, n in enumerate(lengths):
        want = torch.sort(z[off[i]:off[i + 1]], descending=True, stable=True).indices[:k[i]].sort().values
        assert torch.equal(out["kept_idx"][ko[i]:ko[i + 1]].long(), want), i
    assert svl.svl_get_device_status(m.handle) == 0
    m.close()


def test_work_lists_of_many_samples():
    """700 samples of 0 to 3 rows with random gates (several scan chunks, empty samples, one-row runs): every row equals
    the same row of a forward over its 50-sample piece up to bf16 storage (rows are independent; only the K-split of a
    tile may differ)."""
    dims = synth.reduced(TINY.dims, n_layers=3)
    m, _ = _model(dims, 11, max_seq=64)
    g = torch.Generator().manual_seed(12)
    B, L, G, D = 700, dims.n_layers, dims.n_groups, dims.d_model
    n = torch.randint(0, 4, (B,), generator=g)
    lg = (torch.rand(B, L, generator=g) < 0.8).to(torch.uint8)
    gg = (torch.rand(B, L, G, generator=g) < 0.6).to(torch.uint8)
    X0 = torch.randn(int(n.sum()), D, generator=g).to(torch.bfloat16)

    def forward(b0, b1):
        nb, cu = n[b0:b1], torch.zeros(b1 - b0 + 1, dtype=torch.int32)
        cu[1:] = torch.cumsum(nb, 0).to(torch.int32)
        r0, T = int(n[:b0].sum()), int(nb.sum())
        X = X0[r0:r0 + T].cuda()
        pos = torch.cat([torch.arange(int(x)) for x in nb]).to(torch.int32).cuda()
        logits = torch.empty(b1 - b0, dims.vocab, device="cuda")
        ws = torch.empty(svl.svl_workspace_size_for(m.handle, ("prefill",), b1 - b0, T, 0), dtype=torch.uint8,
                         device="cuda")
        svl.svl_gated_prefill(m.handle, b1 - b0, T, X, cu.cuda(), pos, lg[b0:b1].contiguous().cuda(),
                              gg[b0:b1].contiguous().cuda(), svl.SVL_LOGITS_LAST, logits, ws, ws.numel())
        return X

    whole = forward(0, B)
    pieces = torch.cat([forward(i, i + 50) for i in range(0, B, 50)])
    assert svl.svl_get_device_status(m.handle) == 0
    # two bf16 roundings a layer, each at most 2^-9 of a row's largest entries
    assert float((whole.double() - pieces.double()).norm() / pieces.double().norm()) < 2 * L * 2.0 ** -9
    off = torch.repeat_interleave((lg == 0).all(1) | (gg * lg[:, :, None] == 0).all(2).all(1), n)
    assert torch.equal(whole.cpu()[off], X0[off])  # samples with every layer skipped stay as they were
    m.close()


class _Stage:
    """One layer's stages over a packed batch of the given lengths, every group on."""

    def __init__(self, dims, lengths, seed, **kw):
        self.dims = dims
        self.m, self.w = _model(dims, seed, max_seq=4096, **kw)
        B, self.T = len(lengths), sum(lengths)
        self.B, self.cu = B, torch.tensor(np.concatenate([[0], np.cumsum(lengths)]), dtype=torch.int32).cuda()
        self.pos = torch.cat([torch.arange(x) for x in lengths]).to(torch.int32).cuda()
        self.lg = torch.ones(B, 1, dtype=torch.uint8, device="cuda")
        self.gg = torch.ones(B, 1, dims.n_groups, dtype=torch.uint8, device="cuda")
        need = svl.svl_workspace_size_for(self.m.handle, ("prefill",), B, self.T, 0)
        self.ws = torch.empty(need, dtype=torch.uint8, device="cuda")

    def run(self, stage, X, **bufs):
        svl.svl_layer_stage(self.m.handle, stage, 0, self.B, self.T, X, self.cu, self.pos, self.lg, self.gg,
                            workspace=self.ws, workspace_bytes=self.ws.numel(), **bufs)
        torch.cuda.synchronize()
        assert svl.svl_get_device_status(self.m.handle) == 0


def _rand(*shape, seed, std=1.0):
    return (torch.randn(*shape, device="cuda", generator=torch.Generator("cuda").manual_seed(seed)) * std).to(
        torch.bfloat16)


@pytest.mark.parametrize("rows", [1, 32, 33, 100, 300, 515, 1217])
def test_residual_gemms_at_every_kind_of_tail(rows):
    """O and down at LLaVA-7B widths: THIN launches (<= 32 rows, eight shares), three shares of ragged row slices, no
    split, and a split tail after full waves; one bf16 ulp plus the float32 accumulation bound."""
    dims = synth.reduced(LLAVA.dims, n_layers=1, vocab=512)
    s = _Stage(dims, [rows], 21)
    lw = s.w["layers"][0]
    for stage, key, name, width in ((svl.SVL_LAYER_OPROJ, "ao", "wo", dims.d_model),
                                    (svl.SVL_LAYER_DOWN, "h", "wd", dims.d_ffn)):
        X, a = _rand(rows, dims.d_model, seed=22), _rand(rows, width, seed=23, std=0.5)
        ref = X.to(F64) + a.to(F64) @ lw[name].to(F64).T
        bound = ACC * (a.to(F64).abs() @ lw[name].to(F64).abs().T)
        s.run(stage, X, **{key: a})
        check_close(f"{name} {rows}", np64(X), O.round_bf16(np64(ref)), np64(bound))
    s.m.close()


@pytest.mark.parametrize("lengths", [[900, 130, 1500, 40], [769], [768, 768], [300] * 5 + [1]])
def test_attention_items_by_size_and_head_by_head(lengths):
    """Samples over and up to the length from which items are ordered by size: every query block of every head is
    computed once, against softmax attention in float64 (bf16 probabilities: 2^-8 of the weighted |v|)."""
    dims = synth.reduced(synth.WORKLOADS["qwen"].dims, n_layers=1, vocab=512)
    s = _Stage(dims, lengths, 31)
    A, Akv, dh, T = dims.n_heads, dims.n_kv_heads, dims.d_head, s.T
    q, k = _rand(T, A * dh, seed=32), _rand(T, Akv * dh, seed=33)
    vt = _rand(Akv * dh, (T + 7) // 8 * 8, seed=34)
    ao = torch.full((T, A * dh), float("nan"), dtype=torch.bfloat16, device="cuda")
    s.run(svl.SVL_LAYER_ATTN, _rand(T, dims.d_model, seed=35), q=q, k=k, vt=vt, ao=ao)
    r0 = 0
    for n in lengths:
        r = slice(r0, r0 + n)
        mask = torch.ones(n, n, dtype=torch.bool, device="cuda").triu(1)
        for h in range(0, A, 5):
            j = h // (A // Akv)
            sc = q[r, h * dh:(h + 1) * dh].to(F64) @ k[r, j * dh:(j + 1) * dh].to(F64).T / dh ** 0.5
            p = torch.softmax(sc.masked_fill(mask, float("-inf")), -1)
            v = vt[j * dh:(j + 1) * dh, r].to(F64).T
            check_close(f"attn {n} head {h}", np64(ao[r, h * dh:(h + 1) * dh]), O.round_bf16(np64(p @ v)),
                        (2.0 ** -8 * (1 + 1e-3) + ACC) * np64(p @ v.abs()), l2_bar=4e-3)
        r0 += n
    s.m.close()


@pytest.mark.parametrize("heads,kv_heads,n_vis,s_text", [(8, 2, [64, 3], [9, 1]), (20, 2, [40, 120], [5, 30]),
                                                         (8, 2, [1100], [40])])
def test_decode_with_shared_kv_heads(heads, kv_heads, n_vis, s_text):
    """Four and ten query heads per KV head (one and two passes of eight), caches shorter than the eight runs and
    longer than one step of 128 positions per run, against the oracle's forward over the extended prompt."""
    dims = synth.reduced(TINY.dims, n_layers=2, n_heads=heads, n_kv_heads=kv_heads, d_model=64 * heads,
                         c_vis=64 * heads, n_groups=2)
    steps, budgets = 3, [1.0] * len(n_vis)
    case, r = _decode(dims, TINY, 41, n_vis, s_text, budgets, steps, max_len=1200)
    out = r["out"]
    for i in range(len(n_vis)):
        v0, v1 = case.b_np["vis_off"][i], case.b_np["vis_off"][i + 1]
        t0, t1 = case.b_np["text_off"][i], case.b_np["text_off"][i + 1]
        args = (dims, case.w_np, case.b_np["vis"][v0:v1], case.b_np["text_ids"][t0:t1], budgets[i],
                case.b_np["layer_gate"][i], case.b_np["group_gate"][i], r["fed"][:, i].numpy())
        f32, s32 = O.decode_reference(*args, mode="fp32")
        f16, s16 = O.decode_reference(*args, mode="bf16")
        kept = out["kept_idx"][out["kept_off"][i]:out["kept_off"][i + 1]].numpy()
        if not check_selection(out["scores"][v0:v1].numpy(), kept, f32):
            f32, s32 = O.decode_reference(*args, mode="fp32", kept=kept)
            f16, s16 = O.decode_reference(*args, mode="bf16", kept=kept)
        for t in range(steps):
            got = r["logits"][t][i].double().numpy()
            e, bar = rel_err(got, s32[t]["logits"]), bar_for(s32[t], s16[t], "logits")
            assert e < bar, (i, t, e, bar)
            assert int(r["next"][t][i]) == int(np.argmax(r["logits"][t][i].numpy()))
    case.close()


@pytest.mark.parametrize("n_vis,keep", [(1, 1), (128, 128), (300, 129), (576, 289), (3000, 2590)])
def test_projector_tiles(n_vis, keep):
    """Narrow tiles (few rows) and wide ones with a last wave cut into halves, rows that do and do not fill a tile:
    W2 GELU(W1 x) with a bf16 hidden row in float64. Both roundings to bf16 are at most 2^-9 of a value."""
    dims = synth.reduced(LLAVA.dims, n_layers=1, vocab=512)
    m, w = _model(dims, 51, max_seq=4096)
    b = synth.make_batch(LLAVA, 52, n_vis_list=[n_vis], s_text_list=[3], keep_list=[keep], dims=dims, device="cuda")
    out = m.run(b, stages=("select", "pack"))
    assert out["cu_seqlens"].tolist() == [0, keep + 3] and out["pos"][:keep + 3].tolist() == list(range(keep + 3))
    x = b["vis"][out["kept_idx"][:keep].long()].to(F64)
    hid = torch.nn.functional.gelu(x @ w["proj_w1"].to(F64).T).to(torch.bfloat16).to(F64)
    ref = hid @ w["proj_w2"].to(F64).T
    got = out["X"][:keep].to(F64)
    assert float((got - ref).norm() / ref.norm()) < 2 * 2.0 ** -9
    assert torch.equal(out["X"][keep:keep + 3], w["embed"][b["text_ids"].long()])
    assert svl.svl_get_device_status(m.handle) == 0
    m.close()


@pytest.mark.parametrize("fmt", [svl.SVL_GEMM_BF16, svl.SVL_GEMM_E4M3], ids=["bf16", "e4m3"])
@pytest.mark.parametrize("lengths", [[3072], [700, 900, 1, 1500]])
def test_cta_pairs_equal_single_ctas(lengths, fmt, monkeypatch):
    """QKV and gate/up on CTA pairs (the default from 3,072 rows) and on single CTAs: the same bits."""
    dims = synth.reduced(LLAVA.dims, n_layers=1, vocab=512)
    T = sum(lengths)
    got = []
    for env in ("0", None):
        monkeypatch.delenv("SVL_PAIR_GEMM", raising=False)
        if env is not None:
            monkeypatch.setenv("SVL_PAIR_GEMM", env)
        s = _Stage(dims, lengths, 61, gemm_format=fmt)
        X = _rand(T, dims.d_model, seed=62)
        zero = lambda *shape: torch.zeros(*shape, dtype=torch.bfloat16, device="cuda")  # noqa: E731
        q, k, vt, h = zero(T, 4096), zero(T, 4096), zero(4096, (T + 7) // 8 * 8), zero(T, dims.d_ffn)
        s.run(svl.SVL_LAYER_QKV, X, q=q, k=k, vt=vt)
        s.run(svl.SVL_LAYER_GATEUP, X, h=h)
        got.append((q, k, vt, h))
        s.m.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)


def test_e4m3_rows_beyond_one_batch_of_masks():
    """The quantiser's CTAs look the group masks of 128 of their rows up together; 150,000 rows are more than that per
    CTA. Gate/up (gain, equal bits) and down (no gain; its K-split may differ) of the whole against the two halves."""
    dims = synth.reduced(TINY.dims, n_layers=1, vocab=512)
    lengths, half = [500] * 300, 150
    R = 500 * half
    gg = (torch.rand(300, 1, dims.n_groups, generator=torch.Generator().manual_seed(71)) < 0.6).to(torch.uint8).cuda()
    X, h = _rand(2 * R, dims.d_model, seed=72), _rand(2 * R, dims.d_ffn, seed=73)

    def run(s0, s1):
        s = _Stage(dims, lengths[s0:s1], 74, gemm_format=svl.SVL_GEMM_E4M3)
        s.gg = gg[s0:s1].contiguous()
        r = slice(500 * s0, 500 * s1)
        up, out = torch.zeros_like(h[r]), X[r].clone()
        s.run(svl.SVL_LAYER_GATEUP, X[r].contiguous(), h=up)
        s.run(svl.SVL_LAYER_DOWN, out, h=h[r].contiguous())
        s.m.close()
        return up, out

    up, out = run(0, 300)
    a, b = run(0, half), run(half, 300)
    assert torch.equal(up, torch.cat([a[0], b[0]]))
    parts = torch.cat([a[1], b[1]]).double()
    assert float((out.double() - parts).norm() / parts.norm()) < 2.0 ** -9
    src = X[:, :64].contiguous()
    codes, scale = torch.zeros(2 * R, 64, dtype=torch.uint8, device="cuda"), torch.zeros(2 * R, device="cuda")
    pc, ps = torch.zeros_like(codes), torch.zeros_like(scale)
    svl.svl_quantize_rows_e4m3(src, 2 * R, 64, 64, codes, 64, scale)
    for r0 in range(0, 2 * R, 50000):
        svl.svl_quantize_rows_e4m3(src[r0:], 50000, 64, 64, pc[r0:], 64, ps[r0:])
    assert torch.equal(codes, pc) and torch.equal(scale, ps)


@pytest.mark.parametrize("B", [4096, 4500])
def test_pack_of_many_samples(B):
    """Row offsets formed by the gather's own blocks (up to 4,096 samples) and by a launch of their own beyond."""
    m, w = _model(TINY.dims, 81, max_seq=64)
    keep = [(i * 7) % 3 for i in range(B)]
    b = synth.make_batch(TINY, 82, n_vis_list=[2] * B, s_text_list=[1 + i % 2 for i in range(B)], keep_list=keep,
                         device="cuda")
    out = m.run(b, stages=("select", "pack"))
    k, txt = torch.tensor(keep), torch.tensor([1 + i % 2 for i in range(B)])
    assert torch.equal(out["k"].cpu().long(), k)
    cu = torch.cat([torch.zeros(1, dtype=torch.int64), torch.cumsum(k + txt, 0)])
    assert torch.equal(out["cu_seqlens"].cpu().long(), cu)
    T = int(cu[-1])
    within = torch.arange(T) - torch.repeat_interleave(cu[:-1], k + txt)
    assert torch.equal(out["pos"][:T].cpu().long(), within)
    visual = (within < torch.repeat_interleave(k, k + txt)).cuda()
    nk = int(k.sum())
    src = out["kept_idx"][:nk].long() + 2 * torch.repeat_interleave(torch.arange(B), k).cuda()
    assert torch.equal(out["X"][:T][visual], b["vis"][src])
    assert torch.equal(out["X"][:T][~visual], w["embed"][b["text_ids"].long()])
    assert svl.svl_get_device_status(m.handle) == 0
    m.close()


PAIR_DIMS = {"llava": LLAVA.dims, "qwen": synth.WORKLOADS["qwen"].dims, "head64": TINY.dims}


@pytest.mark.parametrize("fmt", [svl.SVL_GEMM_BF16, svl.SVL_GEMM_E4M3], ids=["bf16", "e4m3"])
@pytest.mark.parametrize("lengths", [[1, 129, 255, 257, 40, 3, 128, 300], [33], [384], [60] * 16, [500] * 7],
                         ids=["ragged", "one", "odd", "short", "long"])
@pytest.mark.parametrize("name", list(PAIR_DIMS))
def test_cta_pairs_with_masks(name, lengths, fmt, monkeypatch):
    """Pairs against single CTAs where each sample has group masks of its own (one sample skips the layer): runs that end
    inside a pair, tiles of different runs in one pair, an odd tile without a partner, K and V tiles of one KV head
    (128 or 64 columns). Outputs start as NaN: exactly the active columns are written, with the same bits."""
    dims = synth.reduced(PAIR_DIMS[name], n_layers=1, vocab=512)
    T, B, G = sum(lengths), len(lengths), dims.n_groups
    g = torch.Generator().manual_seed(B + T)
    gg = (torch.rand(B, 1, G, generator=g) < 0.6).to(torch.uint8)
    gg[0] = 1
    if B > 2:
        gg[2] = 0
    on = torch.repeat_interleave(gg[:, 0].bool(), torch.tensor(lengths), 0).cuda()  # [T, G]
    got = []
    for env in ("0", "1"):
        monkeypatch.setenv("SVL_PAIR_GEMM", env)
        s = _Stage(dims, lengths, 65, gemm_format=fmt)
        s.gg = gg.cuda()
        X = _rand(T, dims.d_model, seed=66)
        nan = lambda *shape: torch.full(shape, float("nan"), dtype=torch.bfloat16, device="cuda")  # noqa: E731
        q, k, h = nan(T, dims.n_heads * dims.d_head), nan(T, dims.d_kv), nan(T, dims.d_ffn)
        vt = nan(dims.d_kv, (T + 7) // 8 * 8)
        s.run(svl.SVL_LAYER_QKV, X, q=q, k=k, vt=vt)
        s.run(svl.SVL_LAYER_GATEUP, X, h=h)
        got.append((q, k, vt[:, :T].T, h))
        assert bool(vt[:, T:].isnan().all())
        s.m.close()
    for a, b in zip(*got):
        assert torch.equal(a.contiguous().view(torch.int16), b.contiguous().view(torch.int16))
        assert torch.equal(~b.isnan(), torch.repeat_interleave(on, b.shape[1] // G, 1))

@pytest.mark.parametrize("lengths", [[1000, 1000], [1001, 20], [1001] + [30] * 7, [1001] + [30] * 8])
def test_attention_order_at_the_edges_of_its_rule(lengths):
    """At most eight samples, one of over 1,000 rows: by size; one row fewer or one sample more: head by head."""
    test_attention_items_by_size_and_head_by_head(lengths)


@pytest.mark.parametrize("heads,kv_heads,head_dim", [(28, 4, 128), (32, 4, 64), (20, 2, 64)])
def test_decode_step_of_many_samples_equals_its_samples_alone(heads, kv_heads, head_dim):
    """Grouped KV heads: a batch whose blocks share SMs walks its caches 32 positions a step, a single sample 128; the
    order of every sum is the same, so are the bits. Caches around the eight runs' and the steps' lengths."""
    dims = synth.reduced(synth.WORKLOADS["qwen"].dims, n_layers=1, vocab=512, d_model=heads * head_dim, n_heads=heads,
                         n_kv_heads=kv_heads, d_ffn=1024, c_vis=heads * head_dim, n_groups=2)
    m, _ = _model(dims, 101, max_seq=2048)
    lens = [0, 1, 7, 8, 31, 32, 255, 256, 257, 300, 511, 513, 1023, 1024, 1025, 1500] * 2
    B, max_len, i32 = len(lens), 1600, dict(dtype=torch.int32, device="cuda")
    kv = _rand(2, 1, B, max_len, dims.d_kv, seed=102)

    def step(rows):
        n = len(rows)
        cache = kv[:, :, rows].contiguous()
        tok, length = torch.tensor(rows, **i32), torch.tensor([lens[r] for r in rows], **i32)
        lg = torch.ones(n, 1, dtype=torch.uint8, device="cuda")
        gg = torch.ones(n, 1, dims.n_groups, dtype=torch.uint8, device="cuda")
        logits, nxt = torch.empty(n, dims.vocab, device="cuda"), torch.empty(n, **i32)
        ws = torch.empty(svl.svl_decode_workspace_size(m.handle, n), dtype=torch.uint8, device="cuda")
        svl.svl_decode_step(m.handle, n, tok, cache, max_len, length, lg, gg, logits, nxt, ws, ws.numel())
        assert svl.svl_get_device_status(m.handle) == 0
        return logits, nxt, cache

    whole = step(list(range(B)))
    for r in range(B):
        one = step([r])
        assert torch.equal(whole[0][r], one[0][0]) and torch.equal(whole[2][:, :, r], one[2][:, :, 0]), lens[r]
    m.close()
