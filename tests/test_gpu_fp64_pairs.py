"""The FP64 step of the car grids updates two adjacent headings per thread:
bit for bit against the resident kernel (one quad per thread, the same
per-cell operations) where pairs can go wrong: an odd number of headings, rows
padded by one to three, the smallest axes, negative speeds (the upwind side of
the two lanes differs), and a grid with several pairs per thread."""
import numpy as np
import pytest

from paper_2012_04011_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hj():
    from paper_2012_04011_gb300 import _build
    _build.build()
    from paper_2012_04011_gb300 import hj as mod
    return mod


@pytest.mark.parametrize("n", [(3, 3, 3, 3), (5, 4, 3, 5), (11, 9, 6, 7), (10, 12, 5, 9), (8, 7, 4, 34),
                               (60, 61, 20, 37)])
@pytest.mark.parametrize("lo_v", [0.0, -2.5])
def test_fp64_pairs_equal_resident(hj, n, lo_v):
    lo = (-5.0, -5.0, lo_v, -np.pi)
    grid = scenes.GridSpec(n, lo)
    rng = np.random.default_rng(sum(n))
    V0 = scenes.initial_value(grid, scenes.random_scene(rng, 3)) + 0.1 * rng.standard_normal(n)
    out = []
    for kernel in (hj.HJ_KERNEL_GENERIC, hj.HJ_KERNEL_RESIDENT):
        with hj.Grid(n, lo, grid.hi, grid.periodic, hj.HJ_FP64) as g:
            g.set_dynamics(hj.HJ_DYN_CAR4D, (scenes.A_MAX, scenes.W_MAX))
            g.set_kernel(kernel)
            g.set_initial_value(V0)
            st = g.solve_brt(0.2, scenes.CFL)
            out.append((g.read_value(), st.steps))
    assert out[0][1] == out[1][1] and np.array_equal(out[0][0], out[1][0])
