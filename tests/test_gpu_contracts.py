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
