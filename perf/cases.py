"""Performance cases of the library: what callers run, over the sizes, data types and options they
run it with, each through the public entry points of `paper_2510_22556_b200.binding`.

A case is a plain dict; `kind` names the entry point:

  layer   sablock_compress: one layer of one sequence (a model that compresses layer by layer)
  stack   sablock_compress_layers: every layer of one or more packed sequences in one call
  stages  sablock_segment, _score, _select and _compact one after the other (a caller that looks at
          the scores between them, or pools them)
  decode  sablock_decode_attention: the attention of one decoding step, one call per layer
  host    sablock_compress_layers_host: inputs and outputs in pinned host memory

Inputs are drawn on the GPU from the seed alone: keys with a shared low-rank component (heavy-tailed
attention logits), window queries with a common direction per KV head, a needle span whose keys align
with the mean window query, delimiters at geometric gaps of mean 25 tokens.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2510_22556_b200 import binding as B

VOCAB = 128256
MEAN_GAP = 25
POW2 = "1,2,4,8,16,32"                 # block-size candidates of the 32-row window settings
PAPER = "1,2,3,5,7,9,11,13"            # the paper's own search set (observation window 8)


def _case(**kw):
    c = dict(kind="stack", layers=32, seqs=1, L=131072, L_min=0, len_seed=0, H=32, Hkv=8, D=128, W=32, dtype="bf16",
             budget=1024, candidates=POW2, lse=False, pool=1, pool_mode=0, valid=False)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest call: the fp32 reference-sized prompt, one KV head, everything latency.
        _case(name="tiny_f32", kind="layer", layers=1, L=512, H=4, Hkv=1, D=64, W=16, dtype="f32", budget=64,
              candidates="1,2,4,8"),
        # One Llama-3-8B-shaped layer of an ordinary 8K prompt, compressed right after its own prefill.
        _case(name="layer_8k", kind="layer", layers=1, L=8192, budget=128, candidates="1,2,4,8,16"),
        # The stages called one by one with SnapKV-style pooling, an odd prompt length, window 16.
        _case(name="stages_10k_pool", kind="stages", layers=1, L=9973, W=16, budget=256, candidates="1,2,4,8,16",
              pool=7, pool_mode=0),
        # fp32 cache of the same layer shape (a model served without bf16).
        _case(name="layer_4k_f32", kind="layer", layers=1, L=4096, dtype="f32", budget=256, candidates="1,2,4,8,16"),
        # The paper's own settings: window 8, its search set, a 32-layer stack at 32K.
        _case(name="paper_32k", L=32768, W=8, candidates=PAPER),
        # 32-layer stack at 32K whose prefill hands over its row log-sum-exps.
        _case(name="stack_32k_lse", L=32768, lse=True),
        # Server batch: 16 prompts of 4K to 16K tokens packed together, all layers in one call.
        _case(name="ragged_16", seqs=16, L=16384, L_min=4096, len_seed=4, budget=512, candidates="1,2,4,8,16"),
        # The headline: 128K prompt, 32 layers, the normalisers computed by the pass itself ...
        _case(name="headline_128k"),
        # ... and taken from the prefill.
        _case(name="headline_128k_lse", lse=True),
        # One decoding step over the compacted cache (n_out rows per layer, as compression left them).
        _case(name="decode_1k", kind="decode", L=1024, valid=True),
        # The same step over the full 128K cache.
        _case(name="decode_128k", kind="decode", L=131072),
        # Offloaded cache: inputs and outputs in pinned host memory, the copies part of the call.
        _case(name="host_8k", kind="host", layers=4, L=8192, budget=256, candidates="1,2,4,8,16"),
    ]


def _log_uniform(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choices(["stack", "layer", "f32", "stages", "decode", "host"], [9, 4, 2, 2, 4, 1])[0]
    W = rng.choice([32, 32, 32, 16, 8])
    cands = PAPER if W == 8 else rng.choice([POW2, "1,2,4,8,16"])
    kw = dict(W=W, candidates=cands)

    def budget(L):
        return rng.choice([b for b in (64, 96, 128, 256, 512, 1024, 2048) if b > W and b <= max(L // 2, 64)])

    if what == "stack":
        L = _log_uniform(rng, 1024, 131072)
        seqs = 1 if rng.random() < 0.6 else rng.randint(2, 16)
        while seqs > 1 and seqs * L > 131072:
            seqs = seqs // 2
        layers = rng.choice([8, 16, 32])
        return _case(kind="stack", layers=layers, seqs=seqs, L=L, L_min=max(512, L // 4) if seqs > 1 else 0,
                     len_seed=rng.randint(0, 1 << 20), budget=budget(max(512, L // 4) if seqs > 1 else L),
                     lse=rng.random() < 0.5, **kw)
    if what == "layer":
        L = _log_uniform(rng, 512, 65536)
        return _case(kind="layer", layers=1, L=L, budget=budget(L), lse=rng.random() < 0.3, **kw)
    if what == "f32":
        L = _log_uniform(rng, 256, 8192)
        H, Hkv, D = rng.choice([(4, 1, 64), (32, 8, 128), (8, 8, 64)])
        return _case(kind="layer", layers=1, L=L, H=H, Hkv=Hkv, D=D, dtype="f32", budget=budget(L), **kw)
    if what == "stages":
        L = _log_uniform(rng, 1024, 65536)
        return _case(kind="stages", layers=1, L=L, budget=budget(L), pool=rng.choice([1, 7]), pool_mode=rng.choice([0, 1]),
                     **kw)
    if what == "decode":
        L = _log_uniform(rng, 128, 131072)
        seqs = min(rng.choice([1, 1, 2, 4, 8]), max(1, 131072 // L))
        H, Hkv, D = rng.choice([(32, 8, 128), (32, 8, 128), (32, 32, 128), (16, 8, 64)])
        if H == Hkv:
            L = min(L, 32768)
            seqs = min(seqs, max(1, 32768 // L))
        return _case(kind="decode", layers=rng.choice([8, 32]), seqs=seqs, L=L, H=H, Hkv=Hkv, D=D, valid=L <= 4096)
    L = _log_uniform(rng, 1024, 16384)
    return _case(kind="host", layers=rng.randint(1, 4), L=L, budget=budget(L), **kw)


# ------------------------------------------------------------------------------------- sizes
def _lengths(c):
    if c["seqs"] == 1:
        return [c["L"]]
    r = random.Random(c["len_seed"])
    return [r.randint(c["L_min"], c["L"]) for _ in range(c["seqs"])]


def _offsets(c):
    cu = [0]
    for n in _lengths(c):
        cu.append(cu[-1] + n)
    return cu


def _candidates(c):
    return tuple(int(x) for x in c["candidates"].split(","))


def _dtype(c):
    return torch.float32 if c["dtype"] == "f32" else torch.bfloat16


def work(case):
    """Bytes: keys, queries, token ids (and row log-sum-exps) read once, the retained rows of K and V
    read and written, the index list written.  Operations: the window logits once."""
    c = case
    es = 4 if c["dtype"] == "f32" else 2
    row = c["Hkv"] * c["D"] * es
    nl, ns = c["layers"], c["seqs"]
    if c["kind"] == "decode":
        rows = nl * ns * c["L"]
        return {"bytes": 2 * rows * row + nl * ns * c["H"] * c["D"] * (es + 4), "flops": 4 * rows * c["H"] * c["D"]}
    total = sum(_lengths(c))
    n_out = c["budget"]
    bytes_ = nl * total * row + nl * ns * (c["H"] * c["W"] * c["D"] * es + 4 * n_out * row + 4 * n_out) + 4 * total
    if c["lse"]:
        bytes_ += nl * ns * c["H"] * c["W"] * 4
    if c["kind"] == "stages":                       # seg_id, s, entropy, refined scores out; refined scores in
        bytes_ += 5 * 4 * total
    return {"bytes": bytes_, "flops": 2 * c["H"] * c["W"] * c["D"] * total * nl}


def tolerance(case):
    """Scores and attention outputs are fp32 sums of exactly represented products: 1e-5.  The retained
    rows are copies (compared as whole numbers) and the indices follow from comparisons of fp32
    scores: a pair that is equal to within that rounding may go either way, which moves a few entries
    of one layer's list."""
    return {"rel": 1e-5, "differ": 0.01}


# ------------------------------------------------------------------------------------- inputs
def _bitmap():
    words = torch.zeros((VOCAB + 31) // 32, dtype=torch.int64)
    for i in (VOCAB - 2, VOCAB - 1):
        words[i // 32] |= 1 << (i % 32)
    return torch.where(words >= 2 ** 31, words - 2 ** 32, words).to(torch.int32).cuda()


def _token_ids(L, g):
    ids = torch.randint(0, VOCAB - 2, (L,), generator=g, device="cuda")
    u = torch.rand(max(16, 3 * L // MEAN_GAP + 16), generator=g, device="cuda", dtype=torch.float64).clamp_(1e-12, 1 - 1e-12)
    pos = torch.cumsum(torch.floor(torch.log(u) / math.log(1 - 1 / MEAN_GAP)).to(torch.int64) + 1, 0) - 1
    pos = pos[pos < L]
    para = torch.rand(pos.numel(), generator=g, device="cuda") < 1 / 6
    ids[pos] = VOCAB - 2 + para.to(ids.dtype)
    return ids.to(torch.int32)


def _unit(x):
    return x / x.norm(dim=-1, keepdim=True)


def _keys(L, Hkv, D, g):
    r, kappa = 16, 2.0
    c = torch.randn(L, r, generator=g, device="cuda")
    G = torch.randn(r, Hkv * D, generator=g, device="cuda")
    k = torch.randn(L, Hkv * D, generator=g, device="cuda")
    return k.addmm_(c, G, alpha=kappa / math.sqrt(r)).view(L, Hkv, D)


def _sequence(c, L, g):
    """Window queries [H, W, D] and keys [L, Hkv, D] of one layer of one sequence, in fp32."""
    H, Hkv, D, W = c["H"], c["Hkv"], c["D"], c["W"]
    k = _keys(L, Hkv, D, g)
    u = _unit(torch.randn(Hkv, D, generator=g, device="cuda"))
    q = torch.randn(H, W, D, generator=g, device="cuda") + 3 * u.repeat_interleave(H // Hkv, 0)[:, None]
    n = 24                                                            # the needle
    start = int(0.62 * (L - W - n))
    m = _unit(q.view(Hkv, H // Hkv * W, D).mean(1))
    z = torch.randn(n, Hkv, D, generator=g, device="cuda")
    z = _unit(z - (z * m).sum(-1, keepdim=True) * m)
    k[start:start + n] = math.sqrt(D * 5.0) * (0.9 * m + math.sqrt(1 - 0.81) * z)
    return q, k


def _row_lse(q, k):
    """What a prefill's attention kernel keeps of its last W query rows: the log of the softmax
    normaliser over the causal keys, in fp32."""
    H, W, D = q.shape
    L, Hkv, _ = k.shape
    qf = q.float().view(Hkv, H // Hkv * W, D) / math.sqrt(D)
    x = torch.bmm(qf, k.float().permute(1, 2, 0)).view(Hkv, H // Hkv, W, L)
    hidden = torch.ones(W, W, dtype=torch.bool, device="cuda").triu(1)        # key T + j > query T + w
    x[..., L - W:].masked_fill_(hidden, float("-inf"))
    return torch.logsumexp(x, dim=-1).view(H, W)


def prepare(case, seed):
    c = case
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt, nl, ns = _dtype(c), c["layers"], c["seqs"]
    H, Hkv, D, W = c["H"], c["Hkv"], c["D"], c["W"]
    if c["kind"] == "decode":
        L = c["L"]
        p = B.make_params(H, Hkv, D, W, dt)
        q = torch.randn(nl, ns, H, D, generator=g, device="cuda").to(dt)
        k = torch.empty(nl, ns, L, Hkv, D, dtype=dt, device="cuda")
        v = torch.empty_like(k)
        for i in range(nl):
            for s in range(ns):
                k[i, s] = _keys(L, Hkv, D, g).to(dt)
                v[i, s] = torch.randn(L, Hkv, D, generator=g, device="cuda").to(dt)
        n_valid = torch.full((ns,), L, dtype=torch.int32, device="cuda") if c["valid"] else None
        ws = torch.empty(_decode_ws(p, ns, L), dtype=torch.uint8, device="cuda")
        return dict(c=c, p=p, q=q, k=k, v=v, n_valid=n_valid, ws=ws)

    cu = _offsets(c)
    total, max_L = cu[-1], max(_lengths(c))
    q = torch.empty(nl, ns, H, W, D, dtype=dt, device="cuda")
    k = torch.empty(nl, total, Hkv, D, dtype=dt, device="cuda")
    v = torch.empty_like(k)
    lse = torch.empty(nl, ns, H, W, device="cuda") if c["lse"] else None
    for i in range(nl):
        v[i] = torch.randn(total, Hkv, D, generator=g, device="cuda").to(dt)
        for s in range(ns):
            qs, ks = _sequence(c, cu[s + 1] - cu[s], g)
            q[i, s], k[i, cu[s]:cu[s + 1]] = qs.to(dt), ks.to(dt)
            if lse is not None:
                lse[i, s] = _row_lse(q[i, s], k[i, cu[s]:cu[s + 1]])
    ids = torch.cat([_token_ids(n, g) for n in _lengths(c)])
    kw = dict(pool_kernel=c["pool"], pool_mode=c["pool_mode"])
    if lse is not None:
        kw["row_lse"] = lse
    p = B.make_params(H, Hkv, D, W, dt, _bitmap(), VOCAB, **kw)
    ws = B.alloc_workspace(p, total, max_L, ns, nl)
    st = dict(c=c, p=p, q=q, k=k, v=v, ids=ids, cu=cu, ws=ws, cands=_candidates(c), lse=lse)
    if c["kind"] in ("layer", "stages"):
        st["q"], st["k"], st["v"] = q[0, 0], k[0], v[0]
    if c["kind"] in ("stack", "host"):
        st["out"] = B.LayersOut(p, nl, ns, c["budget"], dt)
    if c["kind"] == "host":
        st["h"] = [x.cpu().pin_memory() for x in (q, k, v, ids)]
        st["h_out"] = B.LayersOut(p, nl, ns, c["budget"], dt, pinned_host=True)
    return st


def _decode_ws(p, n_prob, n_rows):
    import ctypes
    return int(B.lib().sablock_decode_workspace_bytes(ctypes.addressof(p), n_prob, n_rows))


# ------------------------------------------------------------------------------------- one pass
def _bits(x):
    """Copied rows as whole numbers: they are moved, not computed."""
    return x.view(torch.int16 if x.dtype == torch.bfloat16 else torch.int32)


def run(state):
    s, c = state, state["c"]
    p = s["p"]
    if c["kind"] == "layer":
        ok, ov, idx, n = B.compress(p, s["q"], s["k"], s["v"], s["ids"], c["budget"], s["cands"], s["ws"])
        return {"k": _bits(ok), "v": _bits(ov), "idx": idx, "n": n}
    if c["kind"] == "stack":
        o = B.compress_layers(p, s["q"], s["k"], s["v"], s["ids"], s["cu"], c["budget"], s["cands"], s["ws"], s["out"])
        return {"k": _bits(o.out_k), "v": _bits(o.out_v), "idx": o.out_idx, "n": o.n_keep}
    if c["kind"] == "stages":
        seg_id, seg_start, n_seg = B.segment(p, s["ids"], s["ws"])
        sc, ent, ref, _ = B.score(p, s["q"], s["k"], seg_start, n_seg, s["ws"])
        idx, _, _ = B.select(p, ref, c["L"], seg_start, n_seg, c["budget"], s["cands"], s["ws"])
        ok, ov = B.compact(p, s["k"], s["v"], idx)
        return {"seg_id": seg_id, "n_seg": n_seg, "s": sc, "e": ent, "s_refined": ref, "idx": idx, "k": _bits(ok),
                "v": _bits(ov)}
    if c["kind"] == "decode":
        q, k, v, n, ws = s["q"], s["k"], s["v"], s["n_valid"], s["ws"]
        return [B.decode_attention(p, q[i], k[i], v[i], n, ws) for i in range(c["layers"])]
    hq, hk, hv, hi = s["h"]
    h = B.compress_layers_host(p, hq, hk, hv, hi, s["cu"], c["budget"], s["cands"], s["h_out"], s["q"], s["k"], s["v"],
                               s["ids"], s["out"], s["ws"])
    return {"k": _bits(h.out_k), "v": _bits(h.out_v), "idx": h.out_idx, "n": h.n_keep}
