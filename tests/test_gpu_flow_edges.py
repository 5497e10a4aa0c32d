"""The unit-flow score kernel at the edges of its schedule: lengths around a token tile and a unit, every
number of window rows per KV head, long sequences of few window rows, several head groups (more than 1024 window rows:
their sums pass through scratch that has fewer slots than there are problems) in one and two sweeps, packed
sequences of very different length among them ones that are returned unchanged.  Short prompts with one, two, four or eight KV heads take
the pair of kernels of score_pair.cuh in the product, and the same cases are run on the unit flow with a test build that leaves them to
it.  Reference: the scores and entropies in float64 on the stored values.

Tolerance: a logit is an fp32 sum of D <= 128 exact products, partial sums below 64 in log2 units, so its
rounding error is about sqrt(128) * 2^-24 * 64 = 4e-5, times ln 2 the relative error of a weight: 3e-5; the
normaliser adds as much.  Scores: 1e-4 relative.  An entropy is a sum of W terms -a ln a of weights that
carry that error: 2e-4."""
import math

import pytest
import torch

import synth
from paper_2510_22556_b200 import binding as B
from paper_2510_22556_b200.build import build_test_hooks

pytestmark = pytest.mark.gpu


FLOW, PAIR = 2, 3


@pytest.fixture(scope="module")
def hooked():
    return B._load(build_test_hooks())


@pytest.fixture
def on_the_flow(hooked):
    """The test build for the duration of a test, with every call that could take the pair on the unit flow."""
    saved, B._lib = B._lib, hooked
    hooked.sablock_test_no_pair(1)
    yield hooked
    hooked.sablock_test_no_pair(0)
    B._lib = saved


def _kernels(lib, H, Hkv, D, W, lens, n_layers, lse=False):
    p = B.make_params(H, Hkv, D, W, torch.bfloat16, **(dict(row_lse=256) if lse else {}))
    cu = (B.C.c_int * (len(lens) + 1))(0)
    for i, n in enumerate(lens):
        cu[i + 1] = cu[i] + n
    return lib.sablock_test_score_kernels(B.C.c_void_p(B.C.addressof(p)), n_layers, len(lens), cu, max(lens), 64, B.C.c_size_t(1 << 40))


def _reference(q, k, W):
    """q [H, W, D], k [L, Hkv, D] -> s [T], e [T] in float64."""
    H, _, D = q.shape
    L, Hkv, _ = k.shape
    T = L - W
    hidden = torch.ones(W, W, dtype=torch.bool, device=k.device).triu(1)
    abar = torch.zeros(W, L, dtype=torch.float64, device=k.device)
    for j in range(Hkv):
        x = torch.einsum("hwd,ld->hwl", q[j * (H // Hkv):(j + 1) * (H // Hkv)].double(), k[:, j].double()) / math.sqrt(D)
        x[..., T:].masked_fill_(hidden, float("-inf"))
        abar += torch.softmax(x, -1).sum(0)
    a = abar[:, :T]
    hat = a / a.sum(0)
    return a.sum(0) / H, -(hat * torch.log(hat + 1e-6)).sum(0)


def _run(H, Hkv, D, W, lens, n_layers, budget, lse=False):
    cfg = synth.Config("t", n_layers, H, Hkv, D, W, tuple(lens), (budget,), (1, 2, 4), "bf16", 5000, 8, 2.0, 20, (0.4,), 9)
    b = synth.make_batch(cfg, device="cuda")
    kw = dict(row_lse=synth.prefill_row_lse(b.q_win, b.k, b.cu_seqlens)) if lse else {}
    p = B.make_params(H, Hkv, D, W, torch.bfloat16, b.bitmap, cfg.vocab, **kw)
    ws = B.alloc_workspace(p, b.cu_seqlens[-1], max(lens), len(lens), n_layers)
    for rep in range(2):                                         # the second pass finds the first one's scratch
        B.compress_layers(p, b.q_win, b.k, b.v, b.token_ids, b.cu_seqlens, budget, cfg.candidates, ws)
        torch.cuda.synchronize()
        assert B.read_status(ws) == 0
        s = B.workspace_view(p, ws, "s", b.cu_seqlens[-1], max(lens), len(lens), n_layers)
        e = B.workspace_view(p, ws, "e", b.cu_seqlens[-1], max(lens), len(lens), n_layers)
        if rep == 0:
            first = s.clone(), e.clone()
    for l in range(n_layers):
        for i, L in enumerate(lens):
            if L <= budget:
                continue
            a = b.cu_seqlens[i]
            rs, re = _reference(b.q_win[l, i], b.k[l, a:a + L], W)
            ds = (s[l, a:a + L - W].double() - rs).abs() / rs
            assert float(ds.max()) <= 1e-4, (l, i, float(ds.max()))
            assert float((e[l, a:a + L - W].double() - re).abs().max()) <= 2e-4
            assert torch.equal(first[0][l, a:a + L - W], s[l, a:a + L - W])      # fixed summation order
            assert torch.equal(first[1][l, a:a + L - W], e[l, a:a + L - W])


@pytest.mark.parametrize("L", [129, 160, 161, 255, 511, 512, 513, 545, 2047, 2049, 8193])
@pytest.mark.parametrize("lse", [False, True])
def test_lengths(L, lse):
    _run(32, 8, 128, 32, [L], 1, 64, lse)


@pytest.mark.parametrize("L", [129, 160, 161, 255, 511, 512, 513, 545, 2047, 2049, 8193])
@pytest.mark.parametrize("lse", [False, True])
def test_lengths_on_the_flow(on_the_flow, L, lse):
    assert _kernels(on_the_flow, 32, 8, 128, 32, [L], 1, lse) == FLOW
    _run(32, 8, 128, 32, [L], 1, 64, lse)


@pytest.mark.parametrize("H,Hkv,W,D", [(8, 8, 8, 128), (4, 2, 8, 64), (6, 2, 8, 128), (10, 2, 8, 64), (16, 2, 16, 128), (6, 2, 32, 128),
                                       (32, 2, 8, 128), (3, 3, 32, 64), (8, 2, 32, 64), (14, 2, 16, 64)])
@pytest.mark.parametrize("lse", [False, True])
def test_window_rows(H, Hkv, W, D, lse):
    _run(H, Hkv, D, W, [1500], 3, 64, lse)


@pytest.mark.parametrize("H,Hkv,W,D", [(8, 8, 8, 128), (6, 2, 8, 64), (10, 2, 8, 64), (16, 2, 16, 128), (6, 2, 32, 128),
                                       (32, 2, 8, 128), (8, 2, 32, 64), (14, 2, 16, 64), (7, 1, 16, 128), (4, 4, 32, 64)])
@pytest.mark.parametrize("lse", [False, True])
def test_window_rows_on_the_flow(on_the_flow, H, Hkv, W, D, lse):
    assert _kernels(on_the_flow, H, Hkv, D, W, [1500], 3, lse) == FLOW
    _run(H, Hkv, D, W, [1500], 3, 64, lse)


@pytest.mark.parametrize("H,Hkv,W,D,L,n_layers", [(32, 8, 8, 128, 20011, 9), (32, 8, 16, 128, 40000, 6), (16, 4, 8, 64, 70001, 3),     # one group
                                                  (64, 16, 32, 128, 5000, 9), (40, 40, 32, 64, 9001, 6), (35, 35, 32, 128, 2500, 5)])   # two
def test_head_groups(H, Hkv, W, D, L, n_layers):
    _run(H, Hkv, D, W, [L], n_layers, 128)


@pytest.mark.parametrize("H,Hkv,W", [(32, 8, 8), (40, 40, 32), (64, 16, 32)])
def test_head_groups_packed(H, Hkv, W):
    _run(H, Hkv, 128, W, [17000, 300, 60, 9000, 129, 50], 5, 64)


@pytest.mark.parametrize("lse", [False, True])
def test_packed(lse):
    _run(32, 8, 128, 32, [5000, 100, 129, 3333, 64, 700, 1], 12, 64, lse)


@pytest.mark.parametrize("lens,n_layers", [([3000], 6), ([900, 2500, 40], 4)])
def test_single_sweep_with_two_groups(lens, n_layers):
    _run(64, 16, 128, 32, lens, n_layers, 64, True)


@pytest.mark.parametrize("H,Hkv,D,W", [(64, 16, 128, 32),        # two groups of eight heads, 128 window rows each
                                       (35, 35, 64, 32),         # 18 and 17 heads of 32 rows: a smaller last group
                                       (255, 17, 64, 8)])        # 6, 6 and 5 heads of 120 rows: a group between two others
@pytest.mark.parametrize("lens,n_layers", [([3000, 300, 3000], 4),
                                           ([12800] + [129] * 7, 3),
                                           ([700, 40, 2500, 900, 130, 1300], 4)])
@pytest.mark.parametrize("lse", [False, True])
def test_carry_between_head_groups(H, Hkv, D, W, lens, n_layers, lse):
    """More than 1024 window rows: the head groups hand their sums on through scratch that problems of other lengths have
    used before."""
    _run(H, Hkv, D, W, lens, n_layers, 64, lse)


@pytest.mark.parametrize("H,Hkv,D,W", [(32, 8, 128, 32), (8, 2, 64, 8), (6, 2, 128, 16), (64, 16, 64, 32)])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("L", [700, 5000, 9000])
def test_a_key_that_is_no_number(H, Hkv, D, W, value, L):
    """A NaN or infinite element of one key makes the softmax of every window row of its head NaN, and with it all scores, as
    the definition has it; the status word says so."""
    cfg = synth.Config("t", 1, H, Hkv, D, W, (L,), (64,), (1, 2, 4), "bf16", 5000, 8, 2.0, 20, (0.4,), 9)
    b = synth.make_batch(cfg, device="cuda")
    b.k[0, L // 3, 0, 5] = value
    p = B.make_params(H, Hkv, D, W, torch.bfloat16, b.bitmap, cfg.vocab)
    ws = B.alloc_workspace(p, L, L)
    B.compress_layers(p, b.q_win, b.k, b.v, b.token_ids, b.cu_seqlens, 64, cfg.candidates, ws)
    torch.cuda.synchronize()
    rs, _ = _reference(b.q_win[0, 0], b.k[0], W)
    s = B.workspace_view(p, ws, "s", L, L)[0, :L - W]
    assert bool(torch.isnan(rs).all()) and bool(torch.isnan(s).all())
    assert B.read_status(ws) == 6


@pytest.mark.parametrize("H,Hkv,D,W", [(32, 8, 128, 32), (16, 4, 64, 8), (8, 2, 128, 16), (48, 12, 64, 8)])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("L", [700, 5000, 9000])
def test_a_key_that_is_no_number_on_the_flow(on_the_flow, H, Hkv, D, W, value, L):
    assert _kernels(on_the_flow, H, Hkv, D, W, [L], 1) == FLOW
    test_a_key_that_is_no_number(H, Hkv, D, W, value, L)
