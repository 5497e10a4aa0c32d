"""The unit flow's order of units on either side of its rules: units of four tiles that wait where they are, units of one
tile that are put aside, row sums that run ahead by more problems than a call has, by one and by dozens, sequences of very different
length in one period, several head groups.  Reference and tolerances: those of the unit flow's tests."""
import pytest

from test_gpu_flow_edges import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,Hkv,D,W,lens,n_layers", [
    (32, 8, 128, 32, [4096], 16),                                # four tiles a unit, nine problems ahead
    (32, 8, 128, 32, [1500], 32),                                # one tile, dozens of problems ahead
    (32, 8, 128, 8, [700], 40),
    (32, 8, 64, 16, [2214, 553, 900, 60, 1800, 129, 2000, 640, 1111], 6),
    (32, 8, 128, 32, [12000, 200], 4),
    (4, 2, 64, 32, [30000], 2),                                  # two heads: never one tile a unit
    (8, 2, 128, 32, [9000, 300], 12), (12, 3, 128, 32, [6000], 16), (4, 4, 128, 32, [9000], 16), (20, 5, 64, 32, [4096], 16),   # few heads: put aside up to four
    (48, 12, 128, 32, [1300, 40, 2600], 5),                      # two head groups
    (32, 8, 128, 32, [19000], 1)])                               # one problem: nothing to run ahead of
@pytest.mark.parametrize("lse", [False, True])
def test_order_of_units(H, Hkv, D, W, lens, n_layers, lse):
    _run(H, Hkv, D, W, lens, n_layers, 64, lse)
