"""Decode attention at the edges of its launch rules: rows around a 16-row chunk, a 64-row split, the
largest clustered cache and the first one that takes two launches; every head_dim and group size;
problems with few or no valid rows; cache rows that are not contiguous.  Reference: the same
attention in float64 on the stored values.

Tolerance: a logit is an fp32 sum of D <= 256 products, partial sums below 16, so its rounding error is
about sqrt(256) * 2^-24 * 16 = 1.5e-5, which is the relative error of a softmax weight; an output is a
convex combination of rows of V: 2e-5 * max |V|."""
import math

import pytest
import torch

from paper_2510_22556_b200 import binding as B

pytestmark = pytest.mark.gpu


def _reference(q, k, v, n_valid):
    n_prob, H, D = q.shape
    G = H // k.shape[2]
    out = torch.zeros(n_prob, H, D, dtype=torch.float64, device=q.device)
    lse = torch.full((n_prob, H), float("-inf"), dtype=torch.float64, device=q.device)
    for i, n in enumerate(n_valid):
        if n == 0:
            continue
        kk = k[i, :n].double().repeat_interleave(G, 1).permute(1, 0, 2)
        vv = v[i, :n].double().repeat_interleave(G, 1).permute(1, 0, 2)
        x = torch.einsum("hd,hnd->hn", q[i].double(), kk) / math.sqrt(D)
        lse[i] = torch.logsumexp(x, 1)
        out[i] = torch.einsum("hn,hnd->hd", torch.softmax(x, 1), vv)
    return out, lse


@pytest.mark.parametrize("H,Hkv,D,dtype", [(32, 8, 128, torch.bfloat16), (4, 2, 256, torch.bfloat16), (6, 6, 64, torch.bfloat16),
                                           (4, 1, 64, torch.bfloat16), (8, 8, 128, torch.float32)])
@pytest.mark.parametrize("n_rows,n_prob", [(15, 2), (16, 1), (17, 3), (64, 1), (65, 2), (1025, 9), (8192, 1), (8193, 1), (20011, 2)])
def test_decode_edges(H, Hkv, D, dtype, n_rows, n_prob):
    g = torch.Generator(device="cuda").manual_seed(n_rows * 7 + D)
    q = (torch.randn(n_prob, H, D, generator=g, device="cuda") * 1.5).to(dtype)
    k = torch.randn(n_prob, n_rows, Hkv, D, generator=g, device="cuda").to(dtype)
    v = torch.randn(n_prob, n_rows, Hkv, D, generator=g, device="cuda").to(dtype)
    k[0, n_rows // 2] *= 12                                    # a late logit far above the first chunk's maximum
    n_valid = [n_rows if i % 3 == 0 else (0 if i % 3 == 1 else max(1, n_rows - 14)) for i in range(n_prob)]
    p = B.make_params(H, Hkv, D, 8, dtype)
    ref, ref_lse = _reference(q, k, v, n_valid)
    nv = torch.tensor(n_valid, dtype=torch.int32, device="cuda")
    out, lse = B.decode_attention(p, q, k, v, n_valid=nv, want_lse=True)
    tol = 2e-5 * 12 * float(v.double().abs().max())            # the scaled key row has logits twelve times as large
    assert float((out.double() - ref).abs().max()) <= tol
    rows = [i for i, n in enumerate(n_valid) if n]
    assert float((lse.double() - ref_lse)[rows].abs().max()) <= 2e-4
    assert all(bool((lse[i] == float("-inf")).all()) for i, n in enumerate(n_valid) if n == 0)
    assert torch.equal(out, B.decode_attention(p, q, k, v, n_valid=nv))


def test_decode_strided_cache_and_odd_query_address():
    H, Hkv, D, n = 32, 8, 128, 777
    g = torch.Generator(device="cuda").manual_seed(5)
    big = torch.randn(2, n, 2, Hkv, D, generator=g, device="cuda").to(torch.bfloat16)       # K and V interleaved per token
    k, v = big[:, :, 0], big[:, :, 1]
    buf = torch.empty(2 * H * D + 1, dtype=torch.bfloat16, device="cuda")
    q = buf[1:].view(2, H, D)                                                               # two-byte aligned only
    q.copy_(torch.randn(2, H, D, generator=g, device="cuda"))
    st = dict(k_stride_token=2 * Hkv * D, k_stride_layer=n * 2 * Hkv * D, v_stride_token=2 * Hkv * D,
              v_stride_layer=n * 2 * Hkv * D)
    p = B.make_params(H, Hkv, D, 8, torch.bfloat16, **st)
    out = B.decode_attention(p, q, k, v)
    ref, _ = _reference(q, k, v, [n, n])
    assert float((out.double() - ref).abs().max()) <= 2e-5 * float(v.double().abs().max())


@pytest.mark.parametrize("H,Hkv,D", [(8, 2, 128), (4, 4, 64), (4, 2, 256)])
@pytest.mark.parametrize("n_rows", [64, 1024, 20000])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_decode_infinite_values(H, Hkv, D, n_rows, dtype):
    """An infinity in a row of V is one in its column of the output, of its sign, and nowhere else."""
    if dtype == torch.float32:
        D = min(D, 128)
    g = torch.Generator(device="cuda").manual_seed(n_rows + D)
    q = torch.randn(1, H, D, generator=g, device="cuda").to(dtype)
    k, v = (torch.randn(1, n_rows, Hkv, D, generator=g, device="cuda").to(dtype) for _ in range(2))
    v[0, 5, :, 3], v[0, 40, :, 10], v[0, n_rows // 2, :, 33] = float("inf"), float("-inf"), float("inf")
    p = B.make_params(H, Hkv, D, 8, dtype)
    ref, _ = _reference(q, k, v, [n_rows])
    out = B.decode_attention(p, q, k, v).double()
    assert torch.equal(torch.isinf(ref), torch.isinf(out)) and bool((out[torch.isinf(ref)] == ref[torch.isinf(ref)]).all())
    fin = ~torch.isinf(ref)
    assert int(fin.sum()) == H * (D - 3)
    assert float((out - ref)[fin].abs().max()) <= 2e-5 * float(v.double()[torch.isfinite(v)].abs().max())


@pytest.mark.parametrize("H,Hkv,D", [(32, 8, 128), (16, 16, 64), (16, 8, 256)])
@pytest.mark.parametrize("n_rows,n_prob", [(128, 64), (20000, 1)])
def test_decode_values_near_the_end_of_the_range(H, Hkv, D, n_rows, n_prob):
    """Values of 1e38 under logits that rise along the cache: no weight above one, no sum above the largest value."""
    g = torch.Generator(device="cuda").manual_seed(n_rows + D)
    q = torch.randn(n_prob, H, D, generator=g, device="cuda").to(torch.bfloat16)
    k = torch.randn(n_prob, n_rows, Hkv, D, generator=g, device="cuda").to(torch.bfloat16)
    k[:, 64:] += q.view(n_prob, 1, Hkv, H // Hkv, D)[:, :, :, 0] * 0.3                # about 5 in log2 units above the first rows
    v = torch.zeros(n_prob, n_rows, Hkv, D, device="cuda").to(torch.bfloat16)
    v[:, 70] = 1e38
    v[:, n_rows - 3] = -3e37
    p = B.make_params(H, Hkv, D, 8, torch.bfloat16)
    ref, _ = _reference(q, k, v, [n_rows] * n_prob)
    out = B.decode_attention(p, q, k, v).double()
    assert bool(torch.isfinite(out).all())
    assert float((out - ref).abs().max()) <= 2e-5 * 4 * 1e38                        # logits up to four times those above


@pytest.mark.parametrize("H,Hkv,D,n_rows,n_prob", [(32, 8, 128, 6144, 1), (32, 8, 128, 6145, 1), (16, 8, 64, 3072, 1), (16, 8, 64, 3073, 1),
                                                   (32, 8, 128, 9000, 4), (8, 2, 256, 6144, 2), (8, 2, 256, 6145, 2)])
def test_decode_on_either_side_of_the_cluster_rule(H, Hkv, D, n_rows, n_prob):
    """And with a scratch that holds no partial results, which a caller sized for a batch that needs none may bring: the cluster
    takes what it took (8192 rows), longer caches are refused."""
    g = torch.Generator(device="cuda").manual_seed(n_rows + D)
    q = torch.randn(n_prob, H, D, generator=g, device="cuda").to(torch.bfloat16)
    k, v = (torch.randn(n_prob, n_rows, Hkv, D, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    p = B.make_params(H, Hkv, D, 8, torch.bfloat16)
    ref, _ = _reference(q, k, v, [n_rows] * n_prob)
    tol = 2e-5 * float(v.double().abs().max())
    need = int(B.lib().sablock_decode_workspace_bytes(B.C.addressof(p), n_prob, n_rows))
    for nb in {need, 256}:
        ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
        if nb < need and n_rows > 8192:
            with pytest.raises(B.SablockError) as err:
                B.decode_attention(p, q, k, v, ws=ws)
            assert err.value.code == 3
        else:
            assert float((B.decode_attention(p, q, k, v, ws=ws).double() - ref).abs().max()) <= tol
