"""The pass in one call and the same stages called one by one: refined scores and retained positions agree bit for bit
(the stages share their summation orders), for segments of every length around the batches, groups and warps of the
refinement, ranges in shared memory and beyond it, with and without pooling."""
import pytest
import torch

import synth
from paper_2510_22556_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,Hkv,D,W,dtype,L,gap,kw", [
    (32, 8, 128, 32, "bf16", 8192, 25, {}), (32, 8, 128, 32, "bf16", 40000, 25, dict(pool_kernel=7)),
    (4, 1, 64, 16, "f32", 512, 20, {}), (4, 1, 64, 16, "f32", 5000, 3, {}), (8, 2, 64, 8, "f32", 6000, 60, dict(pool_kernel=5, pool_mode=1)),
    (8, 2, 64, 16, "bf16", 30000, 200, {}), (8, 2, 64, 16, "bf16", 30000, 900, {}), (8, 2, 64, 16, "bf16", 30000, 1, {}),
    (4, 1, 64, 8, "bf16", 300000, 25, {}),                       # longer than eight CTAs hold in shared memory
])
def test_stage_by_stage(H, Hkv, D, W, dtype, L, gap, kw):
    cfg = synth.Config("t", 1, H, Hkv, D, W, (L,), (L // 5,), (1, 2, 4, 8), dtype, 5000, 8, 2.0, gap + 1, (0.4,), 3)
    b = synth.make_batch(cfg, device="cuda")
    p = B.make_params(H, Hkv, D, W, synth.torch_dtype(dtype), b.bitmap, cfg.vocab, **kw)
    ws = B.alloc_workspace(p, L, L)
    out = B.compress_layers(p, b.q_win, b.k, b.v, b.token_ids, b.cu_seqlens, L // 5, cfg.candidates, ws)
    torch.cuda.synchronize()
    assert B.read_status(ws) == 0
    fused = {n: B.workspace_view(p, ws, n, L, L)[0, :L - W].clone() for n in ("s", "e", "s_refined")}
    _, seg_start, n_seg = B.segment(p, b.token_ids, ws)
    s, e, sr, _ = B.score(p, b.q_win[0, 0], b.k[0], seg_start, n_seg, ws)
    idx, _, _ = B.select(p, sr, L, seg_start, n_seg, L // 5, cfg.candidates, ws)
    assert torch.equal(s, fused["s"]) and torch.equal(e, fused["e"])
    assert torch.equal(sr, fused["s_refined"])
    assert torch.equal(idx, out.out_idx[0, 0])
