"""Rules that kernels and launches follow, on the CPU: the test build of the library exports the functions
that the device code uses."""
import ctypes as C

import pytest

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
