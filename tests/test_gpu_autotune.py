"""The autotuner's cache: an answer is kept for problems that run the same kernels only."""

import pytest

import paper_2507_23613_gb300 as M
from paper_2507_23613_gb300 import build

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

OMEGA = [6.1, 9.3, 13.0]


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()


@pytest.mark.parametrize("first", [0, 1])
def test_fixed_point_and_fp64_problems_on_one_grid(first):
    """Sides 1 and 20 on equal cells put a coefficient below 2^-10: that problem runs the FP64
    kernels, the square runs in fixed point.  Each is timed for itself, in either order."""
    n = (72 + 8 * first, 72)
    lengths = [(1.0, 1.0), (1.0, 20.0)]
    if first:
        lengths.reverse()
    ms = [M.autotune(n, L, OMEGA)[2] for L in lengths]
    assert ms[0] > 0 and ms[1] > 0 and ms[0] != ms[1]   # (two timings, not one answer twice)
    assert M.autotune(n, lengths[0], OMEGA)[2] == ms[0]


def test_orders_on_one_grid():
    """The answer for the second order (a depth above 1) is none for the fourth."""
    n, L = (72, 64), (1.0, 20.0)
    M.autotune(n, L, OMEGA)
    for length in (L, (1.0, 64 / 72)):
        M.autotune(n, length, OMEGA)
        tb, shape, ms = M.autotune(n, length, OMEGA, order=4)
        assert (tb, shape) == (1, 0) and ms > 0
        M.Solver(n, length, OMEGA, order=4, time_block=tb, tile_shape=shape).close()
