"""The selection kernel where its bookkeeping changes: segments around the longest that one warp
searches, more long segments than its list holds, more segments than shared memory holds starts for, more
segments to search than one round takes, ranges that do not fit shared memory, prompts that get 1, 2,
4 or 8 CTAs, and many problems in one call.  Exact against the oracle (integers)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2510_22556_b200 import binding as B
from test_gpu_stages import _select_case, _sync_ok

pytestmark = pytest.mark.gpu
CANDS = [1, 2, 4, 8, 16, 32]


def _lens(total, draw):
    out, left = [], total
    while left > 0:
        n = min(left, int(draw()))
        out.append(n)
        left -= n
    return np.array(out, np.int64)


@pytest.mark.parametrize("T,lens,B_tok", [
    (1024 * 5, [255, 256, 257, 512] * 4, 1500),                     # around the warp's longest segment
    (60000, [300] * 200, 9000),                                      # two hundred long segments over eight CTAs
    (30000, [400] * 75, 9000),                                       # more of them in a CTA than its list holds
    (9000, [1] * 9000, 700),                                         # more segments than starts in shared memory
    (40000, [4] * 10000, 20000),                                     # thousands of segments to search
    (40000, [30000, 10000], 3000),                                   # ranges of very different length
    (33280 + 1, [33280, 1], 2000),                                   # exactly what shared memory holds, and a token more
    (33281, [33281], 2000),
    (300000, [25] * 12000, 4000),                                    # longer than eight CTAs hold: scores stay in global memory
    (9000, [1023, 1024, 1025, 700, 2], 4000),                        # around the longest segment that a team searches
    (33280, [257] * 129, 20000),                                     # as many of those as a CTA's shared memory holds, in one CTA's share and less
    (450000, [257] * 1750, 90000),                                   # more of them than a CTA's list holds
])
@pytest.mark.parametrize("quantised", [False, True])
def test_select_bookkeeping(T, lens, B_tok, quantised):
    lens = np.array(lens, np.int64)
    if lens.sum() < T:
        rng = np.random.default_rng(T)
        lens = np.concatenate([lens, _lens(T - int(lens.sum()), lambda: rng.geometric(1 / 25.0))])
    _select_case(T, 32, lens, B_tok, CANDS, 0.85, quantised, T + B_tok)


@pytest.mark.parametrize("T", [2, 31, 33, 1023, 2015, 2016, 4063, 4064, 8160, 16352])
def test_select_cluster_sizes(T):
    rng = np.random.default_rng(T)
    _select_case(T, 32, _lens(T, lambda: rng.geometric(1 / 25.0)), max(1, T // 7), CANDS, 0.85, False, T)


@pytest.mark.parametrize("n_layers,L", [(40, 2500), (20, 9001), (150, 700)])
def test_select_many_problems(n_layers, L):
    """One call over many layers: each layer's list equals the oracle's on the library's own scores."""
    cfg = synth.Config("t", n_layers, 8, 2, 64, 16, (L,), (128,), (1, 2, 4, 8), "bf16", 5000, 8, 2.0, 20, (0.4,), 3)
    b = synth.make_batch(cfg, device="cuda")
    p = B.make_params(8, 2, 64, 16, torch.bfloat16, b.bitmap, cfg.vocab)
    ws = B.alloc_workspace(p, L, L, 1, n_layers)
    out = B.compress_layers(p, b.q_win, b.k, b.v, b.token_ids, b.cu_seqlens, 128, cfg.candidates, ws)
    _sync_ok(ws)
    sr = B.workspace_view(p, ws, "s_refined", L, L, 1, n_layers).cpu().numpy()
    ns = int(B.workspace_view(p, ws, "n_seg", L, L, 1, n_layers)[0])
    st = B.workspace_view(p, ws, "seg_start", L, L, 1, n_layers)[: ns + 1].cpu().numpy()
    T = L - 16
    for l in range(0, n_layers, 7):
        r = oracle.select(sr[l, :T].astype(np.float64), st, 112, cfg.candidates, tau=float(np.float32(0.85)))
        assert out.out_idx[l, 0, :112].cpu().numpy().tolist() == r["keep"].tolist()
        assert out.out_idx[l, 0, 112:].cpu().numpy().tolist() == list(range(T, L))


@pytest.mark.parametrize("T,seg,B_tok", [
    (1800, 3, 1500),           # one CTA, 600 segments to search: one round, although a count read late looks like two
    (2014, 2, 2000),           # 1007 of them: a round's list all but full
    (33280, 2, 33000),         # eight CTAs with 2080 each: the list is emptied in between
])
def test_select_counts_the_segments_of_a_round_once(T, seg, B_tok):
    """More than 512 segments to search in a round: whether the list of segments has to be emptied first is decided by
    every thread alike."""
    for rep in range(4):
        _select_case(T, 32, np.full(T // seg, seg, np.int64), B_tok, CANDS, 0.85, False, T + rep)


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("B_tok", [1, 2, 4])
def test_select_sequences_shorter_than_a_cluster(B_tok, order):
    """A few compressible tokens beside a long prompt, whose cluster size they get: most shares are empty."""
    W = 16
    lens = [9000] + [W + t for t in range(2, 10)] + [W + 1, 9000]
    if order:
        lens = lens[1:] + lens[:1]                               # a short sequence comes first in the packed rows
    cfg = synth.Config("t", 2, 8, 2, 64, W, tuple(lens), (W + B_tok,), (1, 2, 4), "bf16", 5000, 8, 2.0, 3, (), 3)
    b = synth.make_batch(cfg, device="cuda")
    p = B.make_params(8, 2, 64, W, torch.bfloat16, b.bitmap, cfg.vocab)
    cu, total = b.cu_seqlens, b.cu_seqlens[-1]
    ws = B.alloc_workspace(p, total, 9000, len(lens), 2)
    ws.fill_(0x7f)                                               # what the pass does not write holds large numbers
    out = B.compress_layers(p, b.q_win, b.k, b.v, b.token_ids, cu, W + B_tok, cfg.candidates, ws)
    _sync_ok(ws)
    sr = B.workspace_view(p, ws, "s_refined", total, 9000, len(lens), 2).cpu().numpy()
    for l in range(2):
        for i, L in enumerate(lens):
            idx = out.out_idx[l, i].cpu().numpy()
            if L <= W + B_tok:
                assert int(out.n_keep[l, i]) == L and idx[:L].tolist() == list(range(L))
                continue
            T = L - W
            _, st = oracle.segment(b.token_ids[cu[i]:cu[i + 1]], W, b.bitmap, cfg.vocab)
            r = oracle.select(sr[l, cu[i]:cu[i] + T].astype(np.float64), st, B_tok, cfg.candidates, tau=float(np.float32(0.85)))
            assert idx[:B_tok].tolist() == r["keep"].tolist() and idx[B_tok:].tolist() == list(range(T, L))


@pytest.mark.parametrize("T,seg", [(640, 4), (20000, 4), (6000, 300), (300000, 25)])
def test_select_reports_scores_that_do_not_order(T, seg):
    """NaN ranks above every number but is no budget: segments whose share of the Top-B is NaN retain nothing, the
    status says so, and the list holds valid positions; beside other numbers a NaN only does not count."""
    W, B_tok = 32, T // 8 // seg * seg
    rng = np.random.default_rng(T)
    sr = rng.random(T).astype(np.float32)
    st = np.arange(0, T + 1, seg).astype(np.int32)
    seg_start = torch.zeros(T + 1, dtype=torch.int32, device="cuda")
    seg_start[: len(st)] = torch.from_numpy(st).cuda()
    n_seg = torch.tensor([len(st) - 1], dtype=torch.int32, device="cuda")
    p = B.make_params(4, 1, 64, W, torch.bfloat16)
    ws = B.alloc_workspace(p, T + W, T + W)

    def run(x):
        idx, g, b = B.select(p, torch.from_numpy(x).cuda(), T + W, seg_start, n_seg, B_tok + W, [1, 2, 4], ws, want_segments=True)
        torch.cuda.synchronize()
        return idx.cpu().numpy(), g.cpu().numpy()[: len(st) - 1], b.cpu().numpy()[: len(st) - 1], B.read_status(ws)

    whole = sr.copy()
    whole[seg: 2 * seg] = np.nan                                 # the second segment
    idx, g, b, status = run(whole)
    assert status == 6 and b[1] == 0 and g[1] == 0 and b.sum() == B_tok - seg
    assert ((idx >= 0) & (idx < T + W)).all() and not ((idx >= seg) & (idx < 2 * seg)).any()
    one = sr.copy()
    one[:seg] = 2.0                                              # a segment that is retained whole ...
    one[1] = np.nan                                              # ... with one NaN in it
    idx, g, b, status = run(one)
    assert status == 0 and b[0] == seg - 1 and b.sum() == B_tok - 1 and idx[:seg].tolist() == list(range(seg))
    idx, g, b, status = run(np.full(T, np.nan, np.float32))
    assert status == 6 and b.sum() == 0 and ((idx >= 0) & (idx < T + W)).all()
