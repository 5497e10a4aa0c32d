"""The fp32 score path on either side of its launch rules: one tile and its remainders, tiles of both sizes,
KV heads spread over clusters of 1 to 8 CTAs, group sizes that do not divide the heads of a thread, odd
windows, rows that only allow scalar loads.  Reference: float64 on the stored values.

Tolerance: a logit is an fp32 sum of D <= 128 rounded products, partial sums below 64 in log2 units: error
about 2 * sqrt(128) * 2^-24 * 64 = 8e-5, times ln 2 the relative error of a weight and as much again of
the normaliser: 1.2e-4; taken as 2e-4 for scores, 4e-4 for entropies."""
import pytest
import torch

import synth
from paper_2510_22556_b200 import binding as B
from test_gpu_flow_edges import _reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,Hkv,D,W,L", [
    (4, 1, 64, 16, 129), (4, 1, 64, 16, 512), (32, 8, 128, 32, 700), (32, 8, 128, 32, 4097), (8, 8, 64, 8, 2500), (6, 2, 32, 5, 333),
    (10, 2, 48, 32, 1000), (3, 3, 128, 1, 200), (2, 1, 128, 64, 900), (16, 8, 64, 7, 6001), (32, 8, 128, 32, 9000),
])
@pytest.mark.parametrize("layers", [1, 5])
def test_fp32_scores(H, Hkv, D, W, L, layers):
    cfg = synth.Config("t", layers, H, Hkv, D, W, (L,), (W + 20,), (1, 2, 4), "f32", 5000, 8, 2.0, 20, (), 3)
    b = synth.make_batch(cfg, device="cuda")
    p = B.make_params(H, Hkv, D, W, torch.float32, b.bitmap, cfg.vocab)
    ws = B.alloc_workspace(p, L, L, 1, layers)
    B.compress_layers(p, b.q_win, b.k, b.v, b.token_ids, b.cu_seqlens, W + 20, cfg.candidates, ws)
    torch.cuda.synchronize()
    assert B.read_status(ws) == 0
    s = B.workspace_view(p, ws, "s", L, L, 1, layers)
    e = B.workspace_view(p, ws, "e", L, L, 1, layers)
    for l in range(layers):
        rs, re = _reference(b.q_win[l, 0], b.k[l], W)
        assert float(((s[l, :L - W].double() - rs).abs() / rs).max()) <= 2e-4
        assert float((e[l, :L - W].double() - re).abs().max()) <= 4e-4


@pytest.mark.parametrize("H,Hkv,D,W", [(16, 8, 256, 8), (4, 4, 256, 4), (6, 2, 256, 1), (8, 8, 128, 1), (8, 2, 128, 2), (8, 2, 128, 4),
                                       (8, 4, 192, 3), (4, 4, 64, 2), (3, 1, 112, 4)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("L,layers", [(9000, 1), (1500, 10)])
@pytest.mark.parametrize("lse", [False, True])
def test_long_rows_and_few_window_positions(H, Hkv, D, W, dtype, L, layers, lse):
    """Shapes whose tile of eight tokens a thread would not fit shared memory."""
    dt = synth.torch_dtype(dtype)
    cfg = synth.Config("t", layers, H, Hkv, D, W, (L,), (W + 20,), (1, 2, 4), dtype, 5000, 8, 2.0, 20, (), 3)
    b = synth.make_batch(cfg, device="cuda")
    kw = dict(row_lse=synth.prefill_row_lse(b.q_win, b.k, b.cu_seqlens)) if lse else {}
    p = B.make_params(H, Hkv, D, W, dt, b.bitmap, cfg.vocab, **kw)
    ws = B.alloc_workspace(p, L, L, 1, layers)
    B.compress_layers(p, b.q_win, b.k, b.v, b.token_ids, b.cu_seqlens, W + 20, cfg.candidates, ws)
    torch.cuda.synchronize()
    assert B.read_status(ws) == 0
    s = B.workspace_view(p, ws, "s", L, L, 1, layers)
    e = B.workspace_view(p, ws, "e", L, L, 1, layers)
    scale = max(1.0, (D / 128) ** 0.5)                           # the bound above grows with the root of D
    for l in range(layers):
        rs, re = _reference(b.q_win[l, 0], b.k[l], W)
        assert float(((s[l, :L - W].double() - rs).abs() / rs).max()) <= 2e-4 * scale
        assert float((e[l, :L - W].double() - re).abs().max()) <= 4e-4 * scale


def test_fp32_unaligned_rows():
    """Keys whose address is a multiple of 4 bytes only."""
    H, Hkv, D, W, L = 8, 2, 64, 16, 777
    g = torch.Generator(device="cuda").manual_seed(1)
    buf = torch.randn(L * Hkv * D + 1, generator=g, device="cuda")
    k = buf[1:].view(L, Hkv, D)
    q = torch.randn(H, W, D, generator=g, device="cuda")
    p = B.make_params(H, Hkv, D, W, torch.float32)
    ws = B.alloc_workspace(p, L, L)
    st = torch.arange(0, L - W + 1, L - W, dtype=torch.int32, device="cuda")
    seg_start = torch.zeros(L - W + 1, dtype=torch.int32, device="cuda")
    seg_start[: st.numel()] = st
    s, e, _, _ = B.score(p, q, k, seg_start, torch.ones(1, dtype=torch.int32, device="cuda"), ws)
    rs, re = _reference(q, k, W)
    assert float(((s.double() - rs).abs() / rs).max()) <= 2e-4 and float((e.double() - re).abs().max()) <= 4e-4


@pytest.mark.parametrize("H,Hkv", [(5, 1), (6, 2), (7, 1), (8, 2)])
@pytest.mark.parametrize("layers,L", [(1, 300), (8, 6000)])
def test_an_infinite_key_under_given_normalisers(H, Hkv, layers, L):
    """Heads that a thread has room for but the KV head has not add nothing, not even where a logit is infinite."""
    D, W = 64, 12
    cfg = synth.Config("t", layers, H, Hkv, D, W, (L,), (W + 20,), (1, 2, 4), "f32", 5000, 8, 2.0, 20, (), 3)
    b = synth.make_batch(cfg, device="cuda")
    lse = synth.prefill_row_lse(b.q_win, b.k, b.cu_seqlens)      # of the keys before one becomes infinite
    t = L // 2
    b.k[:, t, 0, 5] = float("inf")
    b.q_win[..., 5] = b.q_win[..., 5].abs() + 0.1                # every logit of that key is plus infinity
    p = B.make_params(H, Hkv, D, W, torch.float32, b.bitmap, cfg.vocab, row_lse=lse)
    ws = B.alloc_workspace(p, L, L, 1, layers)
    B.compress_layers(p, b.q_win, b.k, b.v, b.token_ids, b.cu_seqlens, W + 20, cfg.candidates, ws)
    torch.cuda.synchronize()
    s = B.workspace_view(p, ws, "s", L, L, 1, layers)[:, :L - W]
    assert bool((s[:, t] == float("inf")).all())
    assert int(torch.isfinite(s).sum()) == s.numel() - layers


@pytest.mark.parametrize("H,Hkv,D,W,L", [
    (4, 1, 64, 16, 129), (4, 1, 64, 16, 512), (32, 8, 128, 32, 700), (32, 8, 128, 32, 4097), (8, 8, 64, 8, 2500), (3, 3, 128, 1, 200),
    (16, 8, 64, 7, 6001), (5, 1, 64, 12, 3000), (6, 2, 128, 25, 900), (7, 1, 64, 16, 400)])
@pytest.mark.parametrize("layers", [1, 5])
@pytest.mark.parametrize("lse", [False, True])
def test_fp32_scores_of_shapes_that_the_tensor_cores_could_take(H, Hkv, D, W, L, layers, lse):
    """(larger calls of these shapes come here by themselves)"""
    cfg = synth.Config("t", layers, H, Hkv, D, W, (L,), (W + 20,), (1, 2, 4), "f32", 5000, 8, 2.0, 20, (), 3)
    b = synth.make_batch(cfg, device="cuda")
    kw = dict(row_lse=synth.prefill_row_lse(b.q_win, b.k, b.cu_seqlens)) if lse else {}
    p = B.make_params(H, Hkv, D, W, torch.float32, b.bitmap, cfg.vocab, score_impl=B.SCORE_SIMT, **kw)
    ws = B.alloc_workspace(p, L, L, 1, layers)
    B.compress_layers(p, b.q_win, b.k, b.v, b.token_ids, b.cu_seqlens, W + 20, cfg.candidates, ws)
    torch.cuda.synchronize()
    assert B.read_status(ws) == 0
    s = B.workspace_view(p, ws, "s", L, L, 1, layers)
    e = B.workspace_view(p, ws, "e", L, L, 1, layers)
    for l in range(layers):
        rs, re = _reference(b.q_win[l, 0], b.k[l], W)
        assert float(((s[l, :L - W].double() - rs).abs() / rs).max()) <= 2e-4
        assert float((e[l, :L - W].double() - re).abs().max()) <= 4e-4


@pytest.mark.parametrize("H,Hkv", [(5, 1), (6, 2), (7, 1), (8, 2)])
@pytest.mark.parametrize("layers,L", [(1, 300), (8, 6000)])
def test_an_infinite_key_under_given_normalisers_on_multiply_adds(monkeypatch, H, Hkv, layers, L):
    """The same where the call is told to take the multiply-adds: the variant of their second pass with absent heads."""
    plain = B.make_params
    monkeypatch.setattr(B, "make_params", lambda *a, **kw: plain(*a, score_impl=B.SCORE_SIMT, **kw))
    test_an_infinite_key_under_given_normalisers(H, Hkv, layers, L)
