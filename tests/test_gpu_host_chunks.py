"""The host-buffer entry point in chunks of layers: calls on either side of the chunk rule, a last chunk that
is smaller, pooling, the row log-sum-exps and pageable buffers; outputs equal to the device call's, and the
intermediate results where the workspace map says they are.  Scores: the chunks may group the row sums
differently from the whole call (fp32 sums of positive terms in another order), 1e-5 relative."""
import threading

import pytest
import torch

import synth
from paper_2510_22556_b200 import binding as B

pytestmark = pytest.mark.gpu


def _case(n_layers, lens, budget=128, pinned=True, lse=False, pool=1, W=32, H=32, impl=B.SCORE_AUTO):
    cfg = synth.Config("t", n_layers, H, 8, 128, W, tuple(lens), (budget,), (1, 2, 4, 8), "bf16", 128256, 16, 2.0, 25, (0.4,), 11)
    b = synth.make_batch(cfg, device="cuda")
    kw = dict(row_lse=synth.prefill_row_lse(b.q_win, b.k, b.cu_seqlens)) if lse else {}
    p = B.make_params(H, 8, 128, W, torch.bfloat16, b.bitmap, cfg.vocab, pool_kernel=pool, score_impl=impl, **kw)
    total, max_L, ns = b.cu_seqlens[-1], max(lens), len(lens)
    ws, ws2 = (B.alloc_workspace(p, total, max_L, ns, n_layers) for _ in range(2))
    ref = B.compress_layers(p, b.q_win, b.k, b.v, b.token_ids, b.cu_seqlens, budget, cfg.candidates, ws2)
    host = [t.cpu().pin_memory() if pinned else t.cpu() for t in (b.q_win, b.k, b.v, b.token_ids)]
    dev = [torch.zeros_like(t) for t in (b.q_win, b.k, b.v, b.token_ids)]
    h_out = B.LayersOut(p, n_layers, ns, budget, torch.bfloat16, pinned_host=True)
    d_out = B.LayersOut(p, n_layers, ns, budget, torch.bfloat16)
    for _ in range(2):
        B.compress_layers_host(p, *host, b.cu_seqlens, budget, cfg.candidates, h_out, *dev, d_out, ws)
    assert B.read_status(ws) == 0
    for name in ("s", "s_refined", "e"):
        x, y = (B.workspace_view(p, w, name, total, max_L, ns, n_layers) for w in (ws, ws2))
        for i, L in enumerate(lens):
            if L > budget:
                a = b.cu_seqlens[i]
                torch.testing.assert_close(x[:, a:a + L - W], y[:, a:a + L - W], rtol=1e-5, atol=1e-5 if name == "e" else 0)
    assert h_out.n_keep.tolist() == ref.n_keep.cpu().tolist()
    diff = sum(int((h_out.out_idx[l, i, :n] != ref.out_idx[l, i, :n].cpu()).sum())
               for l in range(n_layers) for i in range(ns) for n in [int(h_out.n_keep[l, i])])
    assert diff <= 0.001 * h_out.out_idx.numel()                 # a near tie may fall the other way
    for l in range(n_layers):                                    # the rows are the rows of the host's own list
        for i in range(ns):
            n = int(h_out.n_keep[l, i])
            at = (b.cu_seqlens[i] + h_out.out_idx[l, i, :n]).long()
            assert torch.equal(h_out.out_k[l, i, :n], host[1][l, at]) and torch.equal(h_out.out_v[l, i, :n], host[2][l, at])


@pytest.mark.parametrize("n_layers,lens,kw", [
    (1, [8192], {}), (2, [2049], {}), (3, [2049], {}), (4, [8192], {}), (5, [1500], {}), (9, [2100, 300, 100], {}),
    (17, [2500], dict(lse=True)), (4, [4096], dict(pool=7)), (4, [3000], dict(pinned=False)), (6, [5000], dict(W=8)),
    (9, [2100], dict(W=8, H=8)), (9, [2100], dict(W=8, H=8, impl=B.SCORE_TENSOR)),       # a last layer alone would have 64 query rows
])
def test_host_pass_in_chunks(n_layers, lens, kw):
    _case(n_layers, lens, **kw)


@pytest.mark.parametrize("n_layers", [1, 8])
def test_host_pass_that_is_refused_leaves_nothing_in_flight(n_layers):
    """An output address that the gather cannot take shows after the copies and the other stages are enqueued."""
    L, budget = 16384, 128
    cfg = synth.Config("t", n_layers, 32, 8, 128, 32, (L,), (budget,), (1, 2, 4, 8), "bf16", 128256, 16, 2.0, 25, (0.4,), 11)
    b = synth.make_batch(cfg, device="cuda")
    p = B.make_params(32, 8, 128, 32, torch.bfloat16, b.bitmap, cfg.vocab)
    ws = B.alloc_workspace(p, L, L, 1, n_layers)
    host = [t.cpu().pin_memory() for t in (b.q_win, b.k, b.v, b.token_ids)]
    dev = [torch.zeros_like(t) for t in (b.q_win, b.k, b.v, b.token_ids)]
    h_out = B.LayersOut(p, n_layers, 1, budget, torch.bfloat16, pinned_host=True)
    d_out = B.LayersOut(p, n_layers, 1, budget, torch.bfloat16)
    good = d_out.out_k
    d_out.out_k = torch.empty(good.numel() + 1, dtype=good.dtype, device="cuda")[1:]
    torch.cuda.synchronize()
    with pytest.raises(B.SablockError) as err:
        B.compress_layers_host(p, *host, b.cu_seqlens, budget, cfg.candidates, h_out, *dev, d_out, ws)
    assert err.value.code == 2 and torch.cuda.current_stream().query()
    d_out.out_k = good                                           # and the next call is as good as any
    B.compress_layers_host(p, *host, b.cu_seqlens, budget, cfg.candidates, h_out, *dev, d_out, ws)
    assert B.read_status(ws) == 0
    at = h_out.out_idx[:, 0].long()
    for l in range(n_layers):
        assert torch.equal(h_out.out_k[l, 0], host[1][l, at[l]]) and torch.equal(h_out.out_v[l, 0], host[2][l, at[l]])


def test_host_pass_takes_one_profile_slot():
    """Stage times of a call that would go through in chunks: one slot per call, and no stage of it missing."""
    L, n_layers, budget = 8192, 4, 128
    cfg = synth.Config("t", n_layers, 32, 8, 128, 32, (L,), (budget,), (1, 2, 4, 8), "bf16", 128256, 16, 2.0, 25, (0.4,), 11)
    b = synth.make_batch(cfg, device="cuda")
    p = B.make_params(32, 8, 128, 32, torch.bfloat16, b.bitmap, cfg.vocab)
    ws = B.alloc_workspace(p, L, L, 1, n_layers)
    host = [t.cpu().pin_memory() for t in (b.q_win, b.k, b.v, b.token_ids)]
    dev = [torch.zeros_like(t) for t in (b.q_win, b.k, b.v, b.token_ids)]
    h_out = B.LayersOut(p, n_layers, 1, budget, torch.bfloat16, pinned_host=True)
    d_out = B.LayersOut(p, n_layers, 1, budget, torch.bfloat16)
    B.profile_enable(3)
    try:
        for _ in range(2):
            B.compress_layers_host(p, *host, b.cu_seqlens, budget, cfg.candidates, h_out, *dev, d_out, ws)
        used = [B.profile_read(i) for i in range(3)]
    finally:
        B.profile_enable(0)
    assert used[0] and used[1] and not used[2]
    assert all(u[stage] > 0 for u in used[:2] for stage in ("segment", "score_pass1", "search", "compact"))


def test_host_pass_from_several_threads():
    err = []

    def work():
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                _case(4, [4096])
        except Exception as e:                                   # noqa: BLE001
            err.append(e)

    ts = [threading.Thread(target=work) for _ in range(3)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not err, err
