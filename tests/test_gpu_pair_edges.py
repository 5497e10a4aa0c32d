"""The two short-prompt score kernels at the edges of their tiles and of the rule that chooses them: lengths around a tile
and a pair of tiles, one to eight KV heads to a cluster, every number of window rows, packed sequences among them ones that are
returned unchanged, calls on either side of the rule.  Reference and tolerances: those of the unit flow's tests."""
import pytest

from test_gpu_flow_edges import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,Hkv,D,W", [(4, 1, 128, 32), (4, 2, 64, 32), (4, 4, 128, 8), (32, 8, 128, 32), (32, 8, 64, 16), (8, 8, 128, 16),
                                       (6, 2, 128, 8), (7, 1, 64, 16), (10, 2, 64, 8)])
@pytest.mark.parametrize("L", [130, 256, 257, 300, 385, 1024 + 5])
@pytest.mark.parametrize("lse", [False, True])
def test_pair_lengths(H, Hkv, D, W, L, lse):
    _run(H, Hkv, D, W, [L], 1, 64, lse)


@pytest.mark.parametrize("lens,n_layers", [([14080], 1), ([14081], 1), ([9472], 1), ([9473], 1), ([300, 50, 1, 900, 129], 3), ([520] * 12, 1), ([520] * 40, 1)])
@pytest.mark.parametrize("lse", [False, True])
def test_pair_packed_and_its_limit(lens, n_layers, lse):
    _run(32, 8, 128, 32, lens, n_layers, 64, lse)


@pytest.mark.parametrize("H,Hkv,W,lens,n_layers", [(32, 8, 32, [7900], 1), (32, 8, 8, [2000], 4), (32, 8, 32, [13000], 1), (16, 4, 16, [4000, 900], 3),
                                                   (8, 2, 32, [16000], 1)])
@pytest.mark.parametrize("lse", [False, True])
def test_pair_with_rows_of_64_fills_the_device(H, Hkv, W, lens, n_layers, lse):
    """More CTAs than SMs, which the operands alone would let an SM take four of."""
    _run(H, Hkv, 64, W, lens, n_layers, 64, lse)
