"""fp32 scores on the tensor cores, operands split into three bf16 pieces: lengths around a tile and a CTA's share, window rows
that do not fill a product, windows that are no power of two, packed sequences, given log-sum-exps, strided keys, keys that
only the multiply-adds can take, and inputs beyond what the pieces' products can hold.  Reference: float64 on the stored values.

Tolerance: the pieces are exact and what is left out of a product is below 2^-24 of it, so a logit (partial sums below 64 in
log2 units, at most six sums of them in tensor memory) has an error of about 8 * 2^-24 * 64 = 3e-5, times ln 2 the relative error
of a weight and as much again of the normaliser: 4e-5.  Entropies: sums of W terms -a ln a of such weights, 1e-4."""
import pytest
import torch

import synth
from paper_2510_22556_b200 import binding as B
from test_gpu_flow_edges import _reference

pytestmark = pytest.mark.gpu


def _scores(p, b, lens, layers, budget, cands=(1, 2, 4)):
    ws = B.alloc_workspace(p, b.cu_seqlens[-1], max(lens), len(lens), layers)
    B.compress_layers(p, b.q_win, b.k, b.v, b.token_ids, b.cu_seqlens, budget, cands, ws)
    torch.cuda.synchronize()
    return [B.workspace_view(p, ws, n, b.cu_seqlens[-1], max(lens), len(lens), layers) for n in ("s", "e")] + [B.read_status(ws)]


def _batch(H, Hkv, D, W, lens, layers, budget):
    cfg = synth.Config("t", layers, H, Hkv, D, W, tuple(lens), (budget,), (1, 2, 4), "f32", 5000, 8, 2.0, 20, (), 3)
    return cfg, synth.make_batch(cfg, device="cuda")


@pytest.mark.parametrize("H,Hkv,D,W,lens,layers", [
    (4, 1, 64, 16, [127], 1), (4, 1, 64, 16, [128], 1), (4, 1, 64, 16, [129], 1), (4, 1, 128, 32, [145], 1), (4, 1, 128, 32, [256], 1),
    (32, 8, 128, 32, [1025], 1), (32, 8, 128, 32, [8192], 1), (32, 8, 128, 16, [4097], 2), (32, 8, 128, 8, [5000], 1),
    (8, 8, 64, 32, [2500], 3), (8, 8, 64, 8, [777], 2), (6, 2, 128, 5, [1500], 2), (5, 1, 64, 25, [700], 1), (3, 3, 128, 1, [400], 1),
    (16, 2, 64, 12, [300], 9), (32, 8, 128, 32, [700, 40, 129, 1300], 2), (8, 2, 64, 16, [3000, 60, 2000], 5)])
@pytest.mark.parametrize("lse", [False, True])
def test_scores(H, Hkv, D, W, lens, layers, lse):
    cfg, b = _batch(H, Hkv, D, W, lens, layers, W + 20)
    kw = dict(row_lse=synth.prefill_row_lse(b.q_win, b.k, b.cu_seqlens)) if lse else {}
    err = {}
    for impl in (B.SCORE_AUTO, B.SCORE_SIMT):
        p = B.make_params(H, Hkv, D, W, torch.float32, b.bitmap, cfg.vocab, score_impl=impl, **kw)
        s, e, status = _scores(p, b, lens, layers, W + 20)
        assert status == 0
        sq = []
        for l in range(layers):
            for i, L in enumerate(lens):
                if L <= W + 20:
                    continue
                a = b.cu_seqlens[i]
                rs, re = _reference(b.q_win[l, i], b.k[l, a:a + L], W)
                d = (s[l, a:a + L - W].double() - rs) / rs
                if impl == B.SCORE_AUTO:
                    assert float(d.abs().max()) <= 4e-5
                    assert float((e[l, a:a + L - W].double() - re).abs().max()) <= 1e-4
                sq.append(d.pow(2))
        err[impl] = float(torch.cat(sq).mean().sqrt())
    if not lse:                                                  # (given log-sum-exps are fp32: both share their error)
        assert err[B.SCORE_AUTO] <= 1.5 * err[B.SCORE_SIMT] + 1e-7


@pytest.mark.parametrize("H,Hkv,D,W,lens,layers", [(6, 2, 128, 5, [22000], 1), (5, 1, 64, 25, [11000], 1), (16, 2, 64, 12, [700], 10),
                                                   (4, 1, 64, 16, [20001], 1), (3, 3, 128, 1, [26049], 10), (8, 8, 128, 4, [8100, 30], 4)])
def test_given_normalisers_of_calls_large_enough(H, Hkv, D, W, lens, layers):
    """(smaller ones are left to the multiply-adds)"""
    test_scores(H, Hkv, D, W, lens, layers, True)


@pytest.mark.parametrize("offset", [0, 1])
def test_strided_keys(offset):
    """Keys inside a larger buffer, with gaps between heads, tokens and layers; one element further on their rows are not on
    16-byte boundaries and the multiply-adds take them."""
    H, Hkv, D, W, L = 8, 2, 64, 16, 1100
    g = torch.Generator(device="cuda").manual_seed(2)
    buf = torch.randn(L * 400 + 8, generator=g, device="cuda")
    k = torch.as_strided(buf, (L, Hkv, D), (400, 96, 1), offset)
    q = torch.randn(H, W, D, generator=g, device="cuda")
    p = B.make_params(H, Hkv, D, W, torch.float32, k_stride_token=400, k_stride_head=96)
    ws = B.alloc_workspace(p, L, L)
    seg_start = torch.zeros(L - W + 1, dtype=torch.int32, device="cuda")
    seg_start[1] = L - W
    s, e, _, _ = B.score(p, q, k, seg_start, torch.ones(1, dtype=torch.int32, device="cuda"), ws)
    rs, re = _reference(q, k, W)
    assert float(((s.double() - rs).abs() / rs).max()) <= 2e-4 and float((e.double() - re).abs().max()) <= 4e-4


def test_finite_numbers_that_the_pieces_cannot_multiply():
    """A key element whose leading piece rounds to infinity, under a query that is zero there, and a key of minus infinite logits:
    both are ordinary to multiply-adds.  The logits are those of the multiply-adds, the scores those of the reference."""
    H, Hkv, D, W, L = 4, 2, 128, 16, 600
    cfg, b = _batch(H, Hkv, D, W, [L], 1, 64)
    b.q_win[..., 7] = 0.0
    b.k[0, 100, 0, 7] = torch.finfo(torch.float32).max
    b.q_win[..., 9] = b.q_win[..., 9].abs() + 0.1
    b.k[0, 300, 1, 9] = float("-inf")
    p = B.make_params(H, Hkv, D, W, torch.float32, b.bitmap, cfg.vocab)
    s, _, status = _scores(p, b, [L], 1, 64)
    rs, _ = _reference(b.q_win[0, 0], b.k[0], W)
    assert status == 0 and bool(torch.isfinite(rs).all())
    assert float(((s[0, :L - W].double() - rs).abs() / rs.clamp_min(1e-30)).max()) <= 4e-5


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_a_key_that_is_no_number(value):
    H, Hkv, D, W, L = 8, 2, 128, 8, 900
    cfg, b = _batch(H, Hkv, D, W, [L], 1, 64)
    b.k[0, L // 3, 0, 5] = value
    p = B.make_params(H, Hkv, D, W, torch.float32, b.bitmap, cfg.vocab)
    s, _, status = _scores(p, b, [L], 1, 64)
    assert bool(torch.isnan(s[0, :L - W]).all()) and status == 6


@pytest.mark.parametrize("lse", [False, True])
def test_a_workspace_without_room_for_logits(lse):
    """One sized for the multiply-adds, between two guards: the call takes those, and what they compute."""
    H, Hkv, D, W, L = 32, 8, 128, 32, 3000
    cfg, b = _batch(H, Hkv, D, W, [L], 1, 64)
    kw = dict(row_lse=synth.prefill_row_lse(b.q_win, b.k, b.cu_seqlens)) if lse else {}
    plain = B.make_params(H, Hkv, D, W, torch.float32, b.bitmap, cfg.vocab, score_impl=B.SCORE_SIMT, **kw)
    p = B.make_params(H, Hkv, D, W, torch.float32, b.bitmap, cfg.vocab, **kw)
    n = B.workspace_bytes(plain, L, L)
    assert n < B.workspace_bytes(p, L, L)
    buf = torch.full((n + 512,), 0x5a, dtype=torch.uint8, device="cuda")
    res = []
    for q, ws in ((plain, torch.empty(n, dtype=torch.uint8, device="cuda")), (p, buf[256: 256 + n])):
        out = B.compress_layers(q, b.q_win, b.k, b.v, b.token_ids, b.cu_seqlens, 64, cfg.candidates, ws)
        torch.cuda.synchronize()
        assert B.read_status(ws) == 0
        res.append([B.workspace_view(q, ws, x, L, L)[0, :L - W].clone() for x in ("s", "e", "s_refined")] + [out.out_idx, out.out_k])
    assert all(torch.equal(x, y) for x, y in zip(*res))
    assert bool((buf[:256] == 0x5a).all()) and bool((buf[256 + n:] == 0x5a).all())
    with pytest.raises(B.SablockError) as err:
        B.compress_layers(p, b.q_win, b.k, b.v, b.token_ids, b.cu_seqlens, 64, cfg.candidates, buf[256: 255 + n])
    assert err.value.code == 3


@pytest.mark.parametrize("H,Hkv,D,W,lens,layers", [(32, 8, 128, 32, [4096], 1), (4, 1, 64, 16, [512], 1), (8, 2, 128, 8, [16000], 1), (32, 8, 128, 16, [900, 2100], 3)])
def test_the_same_from_run_to_run(H, Hkv, D, W, lens, layers):
    """Whichever CTA of a row block comes last merges the partial sums, in one order."""
    cfg, b = _batch(H, Hkv, D, W, lens, layers, 64)
    p = B.make_params(H, Hkv, D, W, torch.float32, b.bitmap, cfg.vocab)
    first = None
    for _ in range(20):
        s, e, status = _scores(p, b, lens, layers, 64)
        assert status == 0
        res = [torch.cat([x[l, b.cu_seqlens[i]: b.cu_seqlens[i + 1] - W] for l in range(layers) for i in range(len(lens))]) for x in (s, e)]
        if first is None:
            first = [x.clone() for x in res]
        assert torch.equal(first[0], res[0]) and torch.equal(first[1], res[1])


@pytest.mark.parametrize("L", [16384, 16385])
def test_the_largest_call_that_keeps_its_logits(L):
    """64 MB of them, and a token more."""
    H, Hkv, D, W = 32, 8, 128, 32
    cfg, b = _batch(H, Hkv, D, W, [L], 1, 64)
    p = B.make_params(H, Hkv, D, W, torch.float32, b.bitmap, cfg.vocab)
    assert (B.workspace_bytes(p, L, L) > 64 << 20) == (L == 16384)
    s, e, status = _scores(p, b, [L], 1, 64)
    rs, re = _reference(b.q_win[0, 0], b.k[0], W)
    assert status == 0
    assert float(((s[0, :L - W].double() - rs) / rs).abs().max()) <= (4e-5 if L == 16384 else 2e-4)
    assert float((e[0, :L - W].double() - re).abs().max()) <= (1e-4 if L == 16384 else 4e-4)


@pytest.mark.parametrize("H,Hkv,D,W,L", [(32, 8, 128, 32, 256), (32, 8, 128, 32, 1025), (32, 8, 128, 32, 4096), (32, 8, 128, 32, 8192), (4, 1, 64, 16, 512),
                                         (8, 8, 64, 8, 5000), (32, 8, 128, 8, 8192)])
def test_no_further_from_64_bits_than_multiply_adds(H, Hkv, D, W, L):
    """What the file says of its sums: their error is no larger than that of a chain of fp32 multiply-adds, in its root mean square (a twentieth for
    the sample) nor, though tensor memory loses what it drops in one direction, in its mean."""
    cfg, b = _batch(H, Hkv, D, W, [L], 1, 64)
    rs, _ = _reference(b.q_win[0, 0], b.k[0], W)
    rms, mean = {}, {}
    for impl in (B.SCORE_AUTO, B.SCORE_SIMT):
        p = B.make_params(H, Hkv, D, W, torch.float32, b.bitmap, cfg.vocab, score_impl=impl)
        s, _, status = _scores(p, b, [L], 1, 64)
        assert status == 0
        d = (s[0, :L - W].double() - rs) / rs
        rms[impl], mean[impl] = float(d.pow(2).mean().sqrt()), float(d.mean())
    print(f"{H}/{Hkv} {D} W{W} L{L}: rms {rms[B.SCORE_AUTO]:.3g} / {rms[B.SCORE_SIMT]:.3g}, mean {mean[B.SCORE_AUTO]:+.3g} / {mean[B.SCORE_SIMT]:+.3g}")
    assert rms[B.SCORE_AUTO] <= 1.05 * rms[B.SCORE_SIMT]
    assert abs(mean[B.SCORE_AUTO]) <= rms[B.SCORE_SIMT]
