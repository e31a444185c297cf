"""The on-chip form of the resident kernel (FP32 and Q5.27 car grids whose
blocks of columns fit in the SMs' shared memory): bit for bit against the
generic kernel, which evaluates the same per-cell arithmetic, on the sizes
where the blocks can go wrong: blocks one column wide at an end of the grid,
partial blocks, padded theta rows, theta quads with both signs of cos or sin,
negative speeds, V0 that varies within a column, and launches that start from
a step in either buffer."""
import numpy as np
import pytest

from paper_2012_04011_gb300 import scenes

pytestmark = pytest.mark.gpu

STEER = (1.5, np.pi / 18, 0.3)


@pytest.fixture(scope="module")
def hj():
    from paper_2012_04011_gb300 import _build
    _build.build()
    from paper_2012_04011_gb300 import hj as mod
    return mod


def solve(hj, n, prec, kernel, V0, steer=False, chunk=None, lo=scenes.DOMAIN_LO, T=0.4):
    with hj.Grid(n, lo, scenes.DOMAIN_HI, scenes.PERIODIC_THETA, prec) as g:
        if steer:
            g.set_dynamics(hj.HJ_DYN_CAR4D_STEER, STEER)
        else:
            g.set_dynamics(hj.HJ_DYN_CAR4D, (scenes.A_MAX, scenes.W_MAX))
        g.set_kernel(kernel)
        g.set_initial_value(V0)
        total = 0
        while True:
            st = g.advance_brt(T, scenes.CFL, chunk or 1 << 40)
            total += st.steps
            if st.t_final == T:
                break
        return g.read_value(), total


def smooth_v0(n, seed):
    """A V0 that varies along every axis (periodic in theta)."""
    rng = np.random.default_rng(seed)
    x, y, v, th = (np.linspace(0, 1, m, endpoint=d < 3) for d, m in enumerate(n))
    a = rng.uniform(0.5, 1.5, 5)
    return (a[0] * np.cos(5 * x)[:, None, None, None] + a[1] * np.sin(4 * y)[None, :, None, None]
            + a[2] * np.cos(3 * v)[None, None, :, None] * (1 + 0.5 * np.sin(2 * np.pi * th + a[3]))
            + 0.05 * rng.standard_normal(n))


@pytest.mark.parametrize("prec", ["fp32", "q527"])
@pytest.mark.parametrize("n", [(3, 3, 3, 3), (25, 31, 11, 16), (31, 26, 9, 18), (61, 37, 5, 13), (13, 91, 7, 36),
                               (40, 41, 16, 24), (13, 14, 64, 20), (50, 53, 17, 27)])
@pytest.mark.parametrize("flat", [True, False])
def test_onchip_equals_generic(hj, n, prec, flat):
    code = hj.HJ_FP32 if prec == "fp32" else hj.HJ_Q527
    w = scenes.custom_workload(n, n_circles=4, seed=sum(n))
    V0 = scenes.initial_value(w.grid, w.scene) if flat else smooth_v0(n, sum(n))
    for steer, lo in ((False, scenes.DOMAIN_LO), (True, (-5.0, -5.0, -2.0, -np.pi))):
        ref, steps = solve(hj, n, code, hj.HJ_KERNEL_GENERIC, V0, steer, lo=lo)
        for chunk in (None, 2, 3):
            got, s2 = solve(hj, n, code, hj.HJ_KERNEL_RESIDENT, V0, steer, chunk, lo)
            assert s2 == steps and np.array_equal(got, ref), (steer, chunk)


@pytest.mark.parametrize("n4", [16, 32, 48])
@pytest.mark.parametrize("steer", [False, True])
def test_onchip_q527_ignores_weights_of_earlier_dynamics(hj, n4, steer):
    """A call that does not reach its horizon has no cut step and builds no
    table for one: whatever the second weight table holds (here the weights of
    the constant dynamics solved before, nonzero in every lane) takes no part.
    With N4 a multiple of 16 the quad that starts at theta = pi/2 has a lane of
    weight 0 whose cosine (6e-17) differs in sign from the other three's."""
    n = (31, 31, 11, n4)
    w = scenes.custom_workload(n, n_circles=4, seed=3)
    V0 = scenes.initial_value(w.grid, w.scene)
    out = []
    for kernel in (hj.HJ_KERNEL_GENERIC, hj.HJ_KERNEL_RESIDENT):
        with hj.Grid(n, scenes.DOMAIN_LO, scenes.DOMAIN_HI, scenes.PERIODIC_THETA, hj.HJ_Q527) as g:
            g.set_kernel(kernel)
            g.set_dynamics(hj.HJ_DYN_CONST, (1.0, 1.0, 0.0, 0.0))
            g.set_initial_value(V0)
            g.solve_brt(0.4, scenes.CFL)
            if steer:
                g.set_dynamics(hj.HJ_DYN_CAR4D_STEER, STEER)
            else:
                g.set_dynamics(hj.HJ_DYN_CAR4D, (scenes.A_MAX, scenes.W_MAX))
            g.set_initial_value(V0)
            st = g.advance_brt(0.4, scenes.CFL, 3)
            assert st.kernel == kernel and st.steps == 3
            out.append(g.read_value())
    assert np.array_equal(out[0], out[1])
