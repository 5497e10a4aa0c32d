"""Workspaces that start on an 8-byte boundary only (what the widest element of the scratch asks for) give what
aligned ones do, bit for bit, and nothing in front of them or behind them is written."""
import pytest
import torch

import synth
from paper_2510_22556_b200 import binding as B

pytestmark = pytest.mark.gpu


def _offset(ws):
    """The same number of bytes, 8 behind a 256-byte boundary, between two guards."""
    buf = torch.full((ws.numel() + 272,), 0x5a, dtype=torch.uint8, device="cuda")
    assert buf.data_ptr() % 256 == 0
    return buf, buf[8: 8 + ws.numel()]


def _guards_ok(buf, ws):
    torch.cuda.synchronize()
    assert bool((buf[:8] == 0x5a).all()) and bool((buf[8 + ws.numel():] == 0x5a).all())
    assert B.read_status(ws) == 0


@pytest.mark.parametrize("H,Hkv,D,W,dtype,lens", [(8, 2, 64, 16, "f32", [1500]), (32, 8, 128, 32, "bf16", [3000, 40, 700]),
                                                  (40, 40, 64, 32, "bf16", [900, 2000])])
def test_compress_with_an_offset_workspace(H, Hkv, D, W, dtype, lens):
    cfg = synth.Config("t", 3, H, Hkv, D, W, tuple(lens), (64,), (1, 2, 4), dtype, 5000, 8, 2.0, 20, (0.4,), 3)
    b = synth.make_batch(cfg, device="cuda")
    p = B.make_params(H, Hkv, D, W, synth.torch_dtype(dtype), b.bitmap, cfg.vocab)
    args = (p, b.q_win, b.k, b.v, b.token_ids, b.cu_seqlens, 64, cfg.candidates)
    ws = B.alloc_workspace(p, b.cu_seqlens[-1], max(lens), len(lens), 3)
    ref = B.compress_layers(*args, ws)
    buf, off = _offset(ws)
    out = B.compress_layers(*args, off)
    _guards_ok(buf, off)
    for x, y in ((ref.out_k, out.out_k), (ref.out_v, out.out_v), (ref.out_idx, out.out_idx)):
        for i, L in enumerate(lens):
            assert torch.equal(x[:, i, : min(L, 64)], y[:, i, : min(L, 64)])


def test_stages_with_an_offset_workspace():
    H, Hkv, D, W, L = 32, 8, 128, 32, 2500
    cfg = synth.Config("t", 1, H, Hkv, D, W, (L,), (64,), (1, 2, 4), "bf16", 5000, 8, 2.0, 20, (0.4,), 3)
    b = synth.make_batch(cfg, device="cuda")
    p = B.make_params(H, Hkv, D, W, torch.bfloat16, b.bitmap, cfg.vocab)
    ws = B.alloc_workspace(p, L, L)
    buf, off = _offset(ws)
    res = []
    for w in (ws, off):
        seg_id, seg_start, n_seg = B.segment(p, b.token_ids, w)
        s, e, sr, _ = B.score(p, b.q_win[0, 0], b.k[0], seg_start, n_seg, w)
        idx, _, _ = B.select(p, sr, L, seg_start, n_seg, 256, cfg.candidates, w)
        res.append((seg_id, s, e, sr, idx))
    _guards_ok(buf, off)
    assert all(torch.equal(x, y) for x, y in zip(*res))


@pytest.mark.parametrize("n_rows", [500, 20000])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_decode_with_an_offset_workspace(n_rows, dtype):
    H, Hkv, D = 8, 2, 128
    g = torch.Generator(device="cuda").manual_seed(1)
    q = torch.randn(1, H, D, generator=g, device="cuda").to(dtype)
    k, v = (torch.randn(1, n_rows, Hkv, D, generator=g, device="cuda").to(dtype) for _ in range(2))
    p = B.make_params(H, Hkv, D, 8, dtype)
    ref = B.decode_attention(p, q, k, v)
    ws = torch.empty(int(B.lib().sablock_decode_workspace_bytes(B.C.addressof(p), 1, n_rows)), dtype=torch.uint8, device="cuda")
    buf, off = _offset(ws)
    out = B.decode_attention(p, q, k, v, ws=off)
    torch.cuda.synchronize()
    assert torch.equal(out, ref) and bool((buf[:8] == 0x5a).all()) and bool((buf[8 + ws.numel():] == 0x5a).all())
