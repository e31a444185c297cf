"""GPU parity of the Q5.27 fixed-point path (Sec. III-C, Sec. IV-B) against
the fixed-point oracle: integer codes, so every comparison is bit for bit.

Both sides convert V0 with the same rule (nearest, ties to even,
saturating), take the FP64 dt sequence, round the axis weights
dt |xdot_d| / dx_d to 30 fractional bits from the same FP64 product, and
round each Euler increment once, half up.  Full-size grids use sampled
one-step parity from the GPU's own V_n, plus V <= V0 on every cell.
"""
import numpy as np
import pytest

import oracle
from paper_2012_04011_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hj():
    from paper_2012_04011_gb300 import _build
    _build.build()
    from paper_2012_04011_gb300 import hj as mod
    return mod


def oracle_problem(w, dyn=oracle.DYN_CAR4D, params=None):
    if params is None:
        params = (w.a_max, w.w_max)
    return oracle.Problem(w.grid.n, w.grid.lo, w.grid.hi, w.grid.periodic, dyn, params)


def read_codes(g):
    import torch
    out = torch.empty(int(np.prod(g.info().n)), dtype=torch.int32, device="cuda")
    g.read_value_device(out)
    return out.cpu().numpy().reshape(tuple(g.info().n))


def gpu_codes(hj, w, V0, kernel, T=None, dyn=None, params=None):
    with hj.Grid(w.grid.n, w.grid.lo, w.grid.hi, w.grid.periodic, hj.HJ_Q527) as g:
        if dyn is None:
            g.set_dynamics(hj.HJ_DYN_CAR4D, (w.a_max, w.w_max))
        else:
            g.set_dynamics(dyn, params)
        g.set_kernel(kernel)
        g.set_initial_value(V0)
        st = g.solve_brt(w.T if T is None else T, w.cfl)
        return read_codes(g), st, g.read_value()


@pytest.mark.parametrize("kernel", ["generic", "tiled"])
@pytest.mark.parametrize("name", ["car4d_31x31x11x16", "car4d_60x60x20x36"])
def test_q527_solve_bitwise(hj, name, kernel):
    w = scenes.workload(name)
    V0 = scenes.initial_value(w.grid, w.scene)
    Qo, dts = oracle.solve_q527(oracle_problem(w), V0, w.T, w.cfl, nthreads=oracle.max_threads())
    k = hj.HJ_KERNEL_TILED if kernel == "tiled" else hj.HJ_KERNEL_GENERIC
    Q, st, V = gpu_codes(hj, w, V0, k)
    assert st.kernel == k
    assert st.steps == len(dts) and st.dt_first == dts[0] and st.dt_last == dts[-1]
    assert st.t_final == w.T
    assert np.array_equal(Q, Qo), int(np.count_nonzero(Q != Qo))
    assert np.array_equal(V, oracle.from_q527(Qo))  # host readback is exact


SMALL = [(3, 3, 3, 3), (5, 4, 3, 5), (7, 9, 5, 6), (17, 13, 11, 26), (12, 10, 9, 33), (9, 21, 4, 8)]


@pytest.mark.parametrize("n", SMALL)
def test_q527_small_ragged_grids(hj, n):
    w = scenes.custom_workload(n, n_circles=3, n_rects=1, T=0.4, seed=sum(n))
    V0 = scenes.initial_value(w.grid, w.scene)
    Qo, dts = oracle.solve_q527(oracle_problem(w), V0, w.T, w.cfl)
    for k in (hj.HJ_KERNEL_GENERIC, hj.HJ_KERNEL_TILED):
        Q, st, _ = gpu_codes(hj, w, V0, k)
        assert st.steps == len(dts)
        assert np.array_equal(Q, Qo), (k, int(np.count_nonzero(Q != Qo)))


@pytest.mark.parametrize("c", [(0.7, -0.4, 0.3, -0.9), (-1.1, 0.0, 0.5, 0.2), (0.0, 0.0, 0.0, 0.0)])
def test_q527_constant_dynamics(hj, c):
    w = scenes.custom_workload((11, 9, 7, 10), n_circles=3, T=0.6, seed=3)
    V0 = scenes.initial_value(w.grid, w.scene)
    Qo, dts = oracle.solve_q527(oracle_problem(w, oracle.DYN_CONST, c), V0, w.T, w.cfl)
    Q, st, _ = gpu_codes(hj, w, V0, hj.HJ_KERNEL_AUTO, dyn=hj.HJ_DYN_CONST, params=c)
    assert st.steps == len(dts)
    assert np.array_equal(Q, Qo)


def test_q527_all_axes_periodic(hj):
    w = scenes.custom_workload((10, 12, 6, 8), n_circles=3, T=0.5, seed=11)
    w.grid.periodic = 0b1111
    V0 = scenes.initial_value(w.grid, w.scene)
    Qo, dts = oracle.solve_q527(oracle_problem(w), V0, w.T, w.cfl)
    Q, st, _ = gpu_codes(hj, w, V0, hj.HJ_KERNEL_AUTO)
    assert st.kernel != hj.HJ_KERNEL_TILED  # the tiled kernel needs x, y, v not periodic
    assert np.array_equal(Q, Qo)
    Q, st, _ = gpu_codes(hj, w, V0, hj.HJ_KERNEL_GENERIC)
    assert np.array_equal(Q, Qo)


def test_q527_every_tile_shape_gives_identical_codes(hj):
    w = scenes.workload("car4d_60x60x20x36")
    V0 = scenes.initial_value(w.grid, w.scene)
    ref = None
    for shape in ([0, 0, 0, 0], [3, 5, 20, 6], [6, 4, 60, 8], [8, 2, 13, 5]):
        with hj.Grid(w.grid.n, w.grid.lo, w.grid.hi, w.grid.periodic, hj.HJ_Q527) as g:
            g.set_dynamics(hj.HJ_DYN_CAR4D, (w.a_max, w.w_max))
            g.set_kernel(hj.HJ_KERNEL_TILED)
            g.set_tile_shape(shape)
            g.set_initial_value(V0)
            g.solve_brt(0.6, w.cfl)
            Q = read_codes(g)
        if ref is None:
            ref = Q
        assert np.array_equal(Q, ref), shape


def test_q527_ingest_and_readback_conversions(hj):
    import torch
    w = scenes.custom_workload((9, 8, 5, 12), n_circles=2)
    V0 = scenes.initial_value(w.grid, w.scene)
    V0[0, 0, 0, :3] = [1e9, -1e9, 2.5 * oracle.Q527_ULP]  # saturation and a tie
    codes = oracle.to_q527(V0)
    with hj.Grid(w.grid.n, w.grid.lo, w.grid.hi, w.grid.periodic, hj.HJ_Q527) as g:
        g.set_dynamics(hj.HJ_DYN_CAR4D, (w.a_max, w.w_max))
        g.set_initial_value(V0)
        assert np.array_equal(read_codes(g), codes)
        assert np.array_equal(g.read_value(), oracle.from_q527(codes))
        # raw codes in, FP32 out
        dev = torch.from_numpy(codes.ravel().copy()).cuda()
        hj.hj_set_initial_value_device(g.handle, dev)
        assert np.array_equal(read_codes(g), codes)
        f32 = torch.empty(codes.size, dtype=torch.float32, device="cuda")
        g.read_value_device(f32)
        assert np.array_equal(f32.cpu().numpy(), oracle.from_q527(codes).ravel().astype(np.float32))
        # a position-only V0 (replicated over v and theta)
        g.set_initial_value_xy(scenes.signed_distance_xy(w.grid, w.scene))
        xy = np.broadcast_to(scenes.signed_distance_xy(w.grid, w.scene)[:, :, None, None], w.grid.n)
        assert np.array_equal(read_codes(g), oracle.to_q527(xy))
        bad = V0.copy()
        bad[1, 1, 1, 1] = np.inf
        with pytest.raises(hj.HjError) as e:
            g.set_initial_value(bad)
        assert e.value.status == hj.HJ_ERR_INVALID_ARG


def test_q527_error_against_fp64_is_table_one_size(hj):
    """Sec. IV-B reports 1.4e-6..1.8e-6 between the fixed-point FPGA result
    and a 32-bit floating-point toolbox; the Q5.27 solve here stays within
    1e-6 of the FP64 solve on the paper's grid size."""
    w = scenes.workload("car4d_60x60x20x36")
    V0 = scenes.initial_value(w.grid, w.scene)
    _, _, Vq = gpu_codes(hj, w, V0, hj.HJ_KERNEL_TILED)
    with hj.Grid.for_workload(w, hj.HJ_FP64) as g:
        g.set_initial_value(V0)
        g.solve_brt(w.T, w.cfl)
        V64 = g.read_value()
    assert float(np.abs(Vq - V64).max()) < 1e-6


def test_q527_dynamics_change_mid_solve(hj):
    w = scenes.workload("car4d_31x31x11x16")
    V0 = scenes.initial_value(w.grid, w.scene)
    t1, new = 0.37, (2.5, 0.4)
    Q0 = oracle.to_q527(V0)
    Q1, _, _ = oracle.advance_q527(oracle_problem(w), Q0, Q0, 0.0, t1, w.cfl)
    Qo, _, d2 = oracle.advance_q527(oracle_problem(w, params=new), Q0, Q1, t1, w.T, w.cfl)
    for k in (hj.HJ_KERNEL_GENERIC, hj.HJ_KERNEL_TILED):
        with hj.Grid(w.grid.n, w.grid.lo, w.grid.hi, w.grid.periodic, hj.HJ_Q527) as g:
            g.set_dynamics(hj.HJ_DYN_CAR4D, (w.a_max, w.w_max))
            g.set_kernel(k)
            g.set_initial_value(V0)
            g.solve_brt(t1, w.cfl)
            g.set_dynamics(hj.HJ_DYN_CAR4D, new)
            st = g.solve_brt(w.T, w.cfl)
            assert st.steps == len(d2)
            assert np.array_equal(read_codes(g), Qo)


@pytest.mark.slow
def test_q527_full_size_sampled_step_parity(hj):
    """128x128x64x96 in the benchmark's launch configuration (tiled kernel):
    one GPU step from the GPU's V_n equals the oracle's step at sampled cells
    (every face, edge and corner class included); V <= V0 everywhere."""
    w = scenes.workload("car4d_128x128x64x96")
    V0 = scenes.initial_value(w.grid, w.scene)
    P = oracle_problem(w)
    rng = np.random.default_rng(23)
    cells = list(rng.choice(V0.size, 4000, replace=False))
    N = w.grid.n
    for i in (0, 1, N[0] // 2, N[0] - 2, N[0] - 1):
        for j in (0, 1, N[1] - 2, N[1] - 1):
            for k in (0, 1, N[2] // 2, N[2] - 1):
                for l in (0, 1, N[3] - 1):
                    cells.append(((i * N[1] + j) * N[2] + k) * N[3] + l)
    cells = np.unique(np.array(cells, dtype=np.int64))
    with hj.Grid(w.grid.n, w.grid.lo, w.grid.hi, w.grid.periodic, hj.HJ_Q527) as g:
        g.set_dynamics(hj.HJ_DYN_CAR4D, (w.a_max, w.w_max))
        assert g.info().kernel == hj.HJ_KERNEL_TILED
        g.set_initial_value(V0)
        g.autotune(8)  # the benchmark's launch configuration: the autotuned tile
        Q0 = read_codes(g)
        assert np.array_equal(Q0, oracle.to_q527(V0))
        for n_before in (0, 9):
            if n_before:
                g.advance_brt(w.T, w.cfl, n_before)
            Qn = read_codes(g)
            st = g.advance_brt(w.T, w.cfl, 1)
            Qn1 = read_codes(g)
            want = oracle.step_cells_q527(P, Qn, Q0, st.dt_last, cells)
            assert np.array_equal(Qn1.reshape(-1)[cells], want)
            assert np.all(Qn1 <= Q0)
        st = g.solve_brt(w.T, w.cfl)
        assert st.t_final == w.T
        assert np.all(read_codes(g) <= Q0)


@pytest.mark.parametrize("shape", [None, (1, 1, 4, 4), (2, 1, 4, 4), (1, 1, 40, 0), (4, 3, 7, 0)])
def test_q527_items_over_several_rounds(hj, shape):
    """CTAs that take several work items (up to 4950 of them, the order turning
    round every other round, the last round partly filled) write every cell
    once: the codes of the generic kernel, bit for bit."""
    w = scenes.custom_workload((40, 45, 11, 8), 4, T=0.3)
    V0 = scenes.initial_value(w.grid, w.scene)
    Q, st, _ = gpu_codes(hj, w, V0, hj.HJ_KERNEL_GENERIC)
    with hj.Grid.for_workload(w, hj.HJ_Q527) as g:
        g.set_kernel(hj.HJ_KERNEL_TILED)
        if shape is not None:
            g.set_tile_shape(shape)
        g.set_initial_value(V0)
        st_t = g.solve_brt(w.T, w.cfl)
        assert st_t.kernel == hj.HJ_KERNEL_TILED and st_t.steps == st.steps
        assert np.array_equal(read_codes(g), Q)


@pytest.mark.parametrize("prec", ["FP32", "Q527"])
@pytest.mark.parametrize("axis", [0, 1])
def test_tile_shape_given_along_one_axis_is_kept(hj, prec, axis):
    """A request for the rows along y or along v only: that extent is taken, the
    other one chosen, down to tiles of one row (which the automatic choice leaves
    out in fixed point), with the same codes."""
    w = scenes.workload("car4d_31x31x11x16")
    V0 = scenes.initial_value(w.grid, w.scene)
    ref = None
    with hj.Grid.for_workload(w, getattr(hj, "HJ_" + prec)) as g:
        g.set_kernel(hj.HJ_KERNEL_TILED)
        for rows in (0, 1, 2, 3, 5):
            shape = [0, 0, 0, 0]
            shape[axis] = rows
            g.set_tile_shape(shape)
            tile = list(g.info().tile)
            if rows:
                assert tile[axis] == rows and tile[1 - axis] > 1, tile
            g.set_initial_value(V0)
            g.solve_brt(w.T, w.cfl)
            V = g.read_value()
            ref = V if ref is None else ref
            assert np.array_equal(V, ref), tile
