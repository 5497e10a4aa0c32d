"""Rules that kernels and launches follow, on the CPU: the test build of the library exports the functions
that the device code uses."""
import ctypes as C
import threading
import time

import pytest
import torch

from paper_2510_22556_b200 import binding as B
from paper_2510_22556_b200.build import build_test_hooks


@pytest.fixture(scope="module")
def rules():
    return C.CDLL(build_test_hooks())


@pytest.mark.parametrize("lens", [[3000, 300, 3000], [12800, 129, 129, 129, 129, 129, 129, 129], [700, 40, 2500, 900, 130], [5000],
                                  [128 + 32, 129 + 32, 900, 33, 4000, 2000]])
def test_a_carry_slot_is_taken_over_from_the_last_tenant_that_has_the_tile(rules, lens):
    """Problem i of a launch has carry slot i % 4; per tile it takes over from the last earlier problem of that slot
    whose sequence reaches so far."""
    W, n_out, n_layers = 32, 64, 9
    cu = [0]
    for n in lens:
        cu.append(cu[-1] + n)
    arr = (C.c_int * len(cu))(*cu)
    scored = [i for i, n in enumerate(lens) if n > n_out]
    probs = [(layer, i) for layer in range(n_layers) for i in scored]
    last = {}                                                    # (slot, tile) -> problem of the call
    for index, (layer, i) in enumerate(probs):
        for tile in range((lens[i] - W + 127) // 128):
            got = rules.sablock_test_carry_tenant(len(lens), arr, W, n_out, index, tile)
            assert got == last.get((index % 4, tile), -1), (index, tile)
        for tile in range((lens[i] - W + 127) // 128):
            last[index % 4, tile] = layer * len(lens) + i


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("H,Hkv", [(1, 1), (2, 1), (3, 1), (8, 8), (16, 8), (32, 8), (14, 2), (64, 1)])
def test_the_plain_score_passes_fit_shared_memory(rules, dtype, H, Hkv):
    """Every head dimension and window that the parameter check accepts, few and many tiles."""
    p = B.make_params(H, Hkv, 64, 8, dtype)
    p.score_impl = B.SCORE_SIMT
    at = C.c_void_p(C.addressof(p))
    for D in range(4 if dtype == torch.float32 else 8, 257, 4 if dtype == torch.float32 else 8):
        for W in range(1, min(64, 2048 // H) + 1):
            p.head_dim, p.window = D, W
            for L, layers in ((W + 5, 1), (9000, 1), (9000, 32)):
                n = rules.sablock_test_simt_smem(at, L, layers)
                assert 0 < n <= 226 * 1024, (D, W, L, layers, n)


@pytest.mark.parametrize("n_ctas,n_exchanges", [(2, 6), (3, 4)])
def test_an_exchange_is_complete_when_every_cta_has_posted(rules, n_ctas, n_exchanges):
    """Every order in which the posts of a cluster can arrive: a CTA that leaves exchange n does so after all CTAs have posted n.
    A barrier counts arrivals and flips its phase at every n_ctas of them; a wait on a parity ends once the phase of that parity
    is over."""
    where = [divmod(rules.sablock_test_exchange(n), 2) for n in range(n_exchanges)]
    # state: per CTA the exchange it waits for (its post is out); posts under way (exchange, to); arrivals per CTA and barrier
    start = (tuple([0] * n_ctas), frozenset((c, 0, to) for c in range(n_ctas) for to in range(n_ctas)), tuple([(0, 0)] * n_ctas))
    seen, todo = {start}, [start]
    while todo:
        at, flying, got = todo.pop()
        nxt = []
        for post in flying:
            _, n, to = post
            bar = where[n][0]
            g = list(map(list, got))
            g[to][bar] += 1
            nxt.append((at, flying - {post}, tuple(map(tuple, g))))
        for c in range(n_ctas):
            n = at[c]
            if n == n_exchanges:
                continue
            bar, parity = where[n]
            if (got[c][bar] // n_ctas) % 2 != parity:            # the phase with that parity has completed
                assert all(a >= n for a in at) and not any(m == n and to == c for _, m, to in flying), (at, flying, got)
                a2 = tuple(a + 1 if i == c else a for i, a in enumerate(at))
                more = frozenset((c, n + 1, to) for to in range(n_ctas)) if n + 1 < n_exchanges else frozenset()
                nxt.append((a2, flying | more, got))
        for s in nxt:
            if s not in seen:
                seen.add(s)
                todo.append(s)


@pytest.mark.parametrize("impl", [B.SCORE_AUTO, B.SCORE_TENSOR])
@pytest.mark.parametrize("n_layers,lens,H,Hkv,W", [(9, [2100], 8, 8, 8), (9, [2100], 32, 8, 32), (17, [700, 1500], 8, 8, 8),
                                                  (3, [2100], 8, 8, 8), (33, [4100], 8, 8, 8), (5, [4100, 90, 300], 16, 8, 8)])
def test_chunks_of_a_host_pass_run_like_the_whole(rules, impl, n_layers, lens, H, Hkv, W):
    """Either all layers at once or chunks of which each, the last one too, has the 128 query rows that the tensor maps
    need."""
    p = B.make_params(H, Hkv, 128, W, torch.bfloat16, score_impl=impl)
    cu = (C.c_int * (len(lens) + 1))(0)
    for i, n in enumerate(lens):
        cu[i + 1] = cu[i] + n
    per = rules.sablock_test_host_chunk(C.c_void_p(C.addressof(p)), n_layers, len(lens), cu, max(lens), 64)
    assert 1 <= per <= n_layers
    for at in range(0, n_layers, per):
        assert min(per, n_layers - at) * len(lens) * H * W >= 128
    if (H, W) == (32, 32):                                       # the rule itself, where nothing stands against it
        assert per == max((n_layers + 7) // 8, -(-(4 << 20) // (cu[len(lens)] * Hkv * 256)))


def test_a_limit_is_never_lowered_by_another_thread(rules):
    """Two threads raise one kernel's limit of shared memory at the same time, the one that needs less being slower: what each
    was granted holds from then on."""
    now, set_to = [0], []

    @C.CFUNCTYPE(C.c_int, C.c_int)
    def setter(n):
        if n == 50:
            time.sleep(0.2)
        now[0] = n
        set_to.append(n)
        return 0

    threads = [threading.Thread(target=rules.sablock_test_raise_limit, args=(n, setter)) for n in (50, 100)]
    for t in threads:
        t.start()
        time.sleep(0.05)
    for t in threads:
        t.join()
    assert now[0] == 100, set_to
    assert rules.sablock_test_raise_limit(70, setter) == 0 and now[0] == 100
    failing = C.CFUNCTYPE(C.c_int, C.c_int)(lambda n: 1)
    assert rules.sablock_test_raise_limit(200, failing) == 1     # a refusal is passed on and not remembered
    assert rules.sablock_test_raise_limit(200, setter) == 0 and now[0] == 200


@pytest.mark.parametrize("D", [64, 128])
def test_an_sm_takes_no_more_short_prompt_ctas_than_it_has_tensor_memory_for(rules, D):
    """228 KB of shared memory per SM, 1 KB of it for every resident CTA beside what the CTA asks for: as many CTAs as have their
    accumulators fit, and not one more, whatever registers the compiler takes."""
    n, most = rules.sablock_test_pair_smem(D), rules.sablock_test_pair_ctas()
    static = 5120                                                # barriers, row sums, log-sum-exps, sums of a warp: 4.7 KB
    assert most * (n + static + 1024) <= 228 * 1024 < (most + 1) * (n + 1024)


@pytest.mark.parametrize("H,Hkv,D,n_prob,n_rows,two", [
    (16, 8, 64, 1, 3200, False), (16, 8, 64, 1, 8192, False), (16, 8, 64, 3, 8192, False), (4, 1, 64, 1, 8000, False),     # rows of 128 bytes
    (32, 8, 128, 1, 6144, False), (32, 8, 128, 1, 6145, True), (32, 8, 128, 2, 8192, True), (32, 8, 128, 3, 6400, False),
    (32, 8, 128, 3, 8192, False), (4, 1, 128, 9, 8192, True), (4, 1, 128, 10, 8192, False), (4, 1, 128, 15, 8192, False),
    (4, 1, 128, 16, 8192, True), (4, 1, 128, 18, 8192, True), (4, 1, 128, 19, 8192, False),
    (8, 2, 256, 2, 6400, True), (8, 2, 256, 3, 6400, False), (16, 8, 256, 1, 8192, False), (16, 8, 256, 2, 6400, True), (8, 2, 256, 12, 7000, True),
    (32, 8, 128, 1, 8193, True), (16, 8, 64, 1, 8193, True), (32, 8, 128, 4, 16384, False)])
def test_decode_takes_the_form_that_measured_faster(rules, H, Hkv, D, n_prob, n_rows, two):
    """A cluster of eight, or as many splits as two CTAs an SM allow and a second launch."""
    p = B.make_params(H, Hkv, D, 8, torch.bfloat16)
    rules.sablock_test_decode_splits.argtypes = [C.c_void_p, C.c_int, C.c_int, C.c_size_t]
    n = rules.sablock_test_decode_splits(C.addressof(p), n_prob, n_rows, 1 << 30)
    assert n == (min(296 // (Hkv * n_prob), -(-n_rows // 64)) if two else -8)
    if n_rows <= 8192:                                           # and the cluster where there is no scratch for the other form
        assert rules.sablock_test_decode_splits(C.addressof(p), n_prob, n_rows, 256) == -8


def _kernels(rules, dtype, H, Hkv, D, W, lens, layers, lse=False, impl=B.SCORE_AUTO, n_out=64, ws_bytes=1 << 40):
    p = B.make_params(H, Hkv, D, W, dtype, score_impl=impl, **(dict(row_lse=256) if lse else {}))    # (an address that nothing reads)
    cu = (C.c_int * (len(lens) + 1))(0)
    for i, n in enumerate(lens):
        cu[i + 1] = cu[i] + n
    return rules.sablock_test_score_kernels(C.c_void_p(C.addressof(p)), layers, len(lens), cu, max(lens), n_out, C.c_size_t(ws_bytes))


FLOW, PAIR = 2, 3


@pytest.mark.parametrize("H,Hkv,W,L,layers,lse,kernels", [
    (32, 8, 32, 8192, 1, True, PAIR), (32, 8, 32, 8300, 1, True, FLOW), (32, 8, 8, 9196, 1, True, FLOW),                     # one sweep
    (32, 8, 32, 2048, 4, True, PAIR), (32, 8, 32, 2305, 4, True, FLOW), (16, 4, 8, 16384, 1, True, PAIR), (16, 4, 8, 17388, 1, True, FLOW),
    (8, 2, 32, 33000, 1, True, PAIR), (8, 2, 32, 36844, 1, True, FLOW),
    (4, 1, 32, 25000, 1, True, PAIR), (4, 1, 32, 40940, 1, True, FLOW), (16, 1, 8, 40940, 1, True, PAIR),
    (32, 8, 32, 14080, 1, False, PAIR), (32, 8, 32, 14081, 1, False, FLOW), (32, 8, 8, 14080, 1, False, PAIR),               # two sweeps
    (16, 8, 32, 14000, 1, False, FLOW), (8, 8, 32, 7600, 1, True, PAIR), (8, 8, 32, 8192, 1, True, FLOW), (8, 8, 32, 8192, 1, False, PAIR), (8, 8, 32, 9196, 1, False, FLOW), (16, 4, 32, 28000, 1, False, PAIR), (16, 4, 8, 18412, 1, False, FLOW),
    (16, 4, 8, 16384, 1, False, PAIR), (8, 2, 32, 37800, 1, False, PAIR), (8, 2, 32, 40940, 1, False, FLOW),
    (4, 1, 32, 36000, 1, False, PAIR), (4, 1, 32, 40940, 1, False, FLOW), (4, 1, 32, 15000, 4, False, PAIR), (4, 1, 32, 30000, 2, False, FLOW)])
def test_short_prompts_take_the_kernels_that_measured_faster(rules, H, Hkv, W, L, layers, lse, kernels):
    assert _kernels(rules, torch.bfloat16, H, Hkv, 128, W, [L], layers, lse) == kernels


@pytest.mark.parametrize("one_tile,group_heads,aside", [(0, 1, 2), (0, 2, 2), (0, 3, 2), (0, 4, 2), (0, 5, 0), (0, 8, 0), (0, 18, 0), (1, 4, 2), (1, 8, 2), (1, 16, 2)])
def test_units_are_put_aside_where_they_are_short(rules, one_tile, group_heads, aside):
    assert rules.sablock_test_flow_aside(one_tile, group_heads) == aside


SIMT, X3 = 0, 1


@pytest.mark.parametrize("H,Hkv,D,W,L,layers,lse,kernels", [
    (32, 8, 128, 32, 300, 1, True, SIMT), (32, 8, 128, 32, 700, 1, True, X3), (32, 8, 128, 16, 700, 1, True, SIMT), (32, 8, 128, 16, 1500, 1, True, X3),
    (32, 8, 128, 8, 1500, 1, True, SIMT), (32, 8, 128, 8, 1500, 3, True, X3), (4, 1, 64, 16, 512, 1, True, SIMT), (8, 8, 128, 32, 3000, 1, True, SIMT),
    (8, 8, 128, 32, 5000, 1, True, X3), (4, 1, 64, 16, 512, 1, False, X3), (32, 8, 128, 32, 300, 1, False, X3), (1, 1, 64, 1, 200, 1, False, X3),
    (32, 8, 128, 32, 16384, 1, False, X3), (32, 8, 128, 32, 16385, 1, False, SIMT), (32, 8, 128, 32, 4096, 4, False, X3),     # 64 MB of logits
    (32, 8, 128, 32, 4096, 5, False, SIMT)])
def test_fp32_scores_take_the_kernels_that_measured_faster(rules, H, Hkv, D, W, L, layers, lse, kernels):
    assert _kernels(rules, torch.float32, H, Hkv, D, W, [L], layers, lse) == kernels


def _scratch(rules, dtype, H, Hkv, D, W, L, layers, impl=B.SCORE_AUTO):
    p = B.make_params(H, Hkv, D, W, dtype, score_impl=impl)
    rules.sablock_workspace_bytes.restype = C.c_size_t
    return rules.sablock_workspace_bytes(C.c_void_p(C.addressof(p)), C.c_longlong(L), L, 1, layers)


@pytest.mark.parametrize("H,Hkv,D,W", [(32, 8, 128, 32), (4, 1, 64, 16), (8, 8, 64, 8)])
def test_scratch_for_logits_is_that_of_calls_which_have_them(rules, H, Hkv, D, W):
    """A call that is too large for kept logits needs what it needs on the multiply-adds, and its workspace, or one sized for
    those, is good for smaller calls too: they then take the multiply-adds themselves."""
    f32 = torch.float32
    for L, layers in ((131072, 1), (4096, 32), (16384, 40)):
        if _kernels(rules, f32, H, Hkv, D, W, [L], layers) == SIMT:
            assert _scratch(rules, f32, H, Hkv, D, W, L, layers) == _scratch(rules, f32, H, Hkv, D, W, L, layers, B.SCORE_SIMT)
    for L in (200, 259, 312, 1000, 4096):
        full, plain = (_scratch(rules, f32, H, Hkv, D, W, L, 1, impl) for impl in (B.SCORE_AUTO, B.SCORE_SIMT))
        logits = H * W * -(-L // 128) * 128 * 4
        assert plain < full and logits <= full - plain + 512 * 1024          # (the partial row sums are smaller or larger by some)
        assert _kernels(rules, f32, H, Hkv, D, W, [L], 1, ws_bytes=full) == X3
        assert _kernels(rules, f32, H, Hkv, D, W, [L], 1, ws_bytes=full - 1) == SIMT
        assert _kernels(rules, f32, H, Hkv, D, W, [L], 1, ws_bytes=plain) == SIMT
        assert _kernels(rules, f32, H, Hkv, D, W, [L], 1, ws_bytes=plain - 1) == -1
    assert _kernels(rules, f32, H, Hkv, D, W, [259], 1, ws_bytes=_scratch(rules, f32, H, Hkv, D, W, 312, 1)) >= 0


@pytest.mark.parametrize("dtype,H,Hkv,D,W,lens,layers,lse", [
    (torch.bfloat16, 32, 8, 128, 32, [8192], 4, False), (torch.bfloat16, 32, 8, 128, 32, [8192], 4, True), (torch.bfloat16, 32, 8, 128, 8, [2500], 9, False),
    (torch.bfloat16, 4, 1, 64, 16, [30000], 9, False), (torch.bfloat16, 32, 8, 128, 32, [2048], 4, False), (torch.bfloat16, 32, 8, 128, 32, [3000, 100], 20, True),
    (torch.float32, 32, 8, 128, 32, [4096], 5, False), (torch.float32, 32, 8, 128, 32, [4096], 4, False), (torch.float32, 32, 8, 128, 16, [700], 4, True)])
def test_layers_of_a_host_pass_take_the_kernels_of_the_whole_call(rules, dtype, H, Hkv, D, W, lens, layers, lse):
    """A few layers alone would take other kernels than all of them.  Inside the whole call they take its own, or are no chunk of it (-1:
    they would not fit its workspace)."""
    p = B.make_params(H, Hkv, D, W, dtype, **(dict(row_lse=256) if lse else {}))
    cu = (C.c_int * (len(lens) + 1))(0)
    for i, n in enumerate(lens):
        cu[i + 1] = cu[i] + n
    whole = _kernels(rules, dtype, H, Hkv, D, W, lens, layers, lse)
    at = C.c_void_p(C.addressof(p))
    for some in range(1, layers):
        assert rules.sablock_test_chunk_kernels(at, layers, len(lens), cu, max(lens), 64, some) in (whole, -1)
    per = rules.sablock_test_host_chunk(at, layers, len(lens), cu, max(lens), 64)
    assert rules.sablock_test_chunk_kernels(at, layers, len(lens), cu, max(lens), 64, per) == whole
