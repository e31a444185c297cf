"""Calls that fail leave a grid as it was, or say that its value is gone: a
call on a stream that is being captured, a step launch that fails (on the
host: no kernel of it runs), a step that timed out (only the flags such a step
leaves; no wait runs out)."""
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


def refused_in_capture(hj, torch, stream, call):
    """call() while the stream is being captured: refused, and nothing captured."""
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        graph.capture_begin(capture_error_mode="relaxed")
        try:
            with pytest.raises(hj.HjError) as e:
                call()
            assert e.value.status == hj.HJ_ERR_CUDA
        finally:
            graph.capture_end()


@pytest.mark.filterwarnings("ignore:The CUDA Graph is empty")
@pytest.mark.parametrize("prec, kernel", [("FP64", "GENERIC"), ("FP32", "TILED"), ("FP32", "RESIDENT"),
                                          ("Q527", "RESIDENT")])
def test_call_on_a_captured_stream_changes_nothing(hj, prec, kernel):
    import torch
    w = scenes.workload("car4d_31x31x11x16")
    V0 = scenes.initial_value(w.grid, w.scene)
    xy = scenes.signed_distance_xy(w.grid, w.scene)
    dev, xy_dev = torch.from_numpy(V0).cuda(), torch.from_numpy(xy.ravel().copy()).cuda()
    code, kern = getattr(hj, "HJ_" + prec), getattr(hj, "HJ_KERNEL_" + kernel)
    with hj.Grid.for_workload(w, code) as g:
        g.set_kernel(kern)
        g.set_initial_value(V0)
        g.solve_brt(w.T, w.cfl)
        ref = g.read_value()
    s = torch.cuda.Stream()
    with hj.Grid.for_workload(w, code, cuda_stream=s.cuda_stream) as g:
        g.set_kernel(kern)
        g.set_initial_value(V0)
        # a first solve of a captured stream must not pass for one that ran
        refused_in_capture(hj, torch, s, lambda: g.solve_brt(w.T, w.cfl))
        if kernel == "TILED":
            refused_in_capture(hj, torch, s, lambda: g.autotune(1))
        st = g.advance_brt(w.T, w.cfl, 5)
        assert st.total_steps == 5
        v5 = g.read_value()
        for call in (lambda: g.set_initial_value(V0), lambda: g.set_initial_value(dev),
                     lambda: g.set_initial_value_xy(xy), lambda: hj.hj_set_initial_value_xy_device(g.handle, xy_dev),
                     lambda: g.advance_brt(w.T, w.cfl, 3), lambda: g.solve_converged(1e-3, w.T, w.cfl)):
            refused_in_capture(hj, torch, s, call)
            info = g.info()
            assert info.total_steps == 5 and info.t == st.t_final
            assert np.array_equal(g.read_value(), v5)
        g.solve_brt(w.T, w.cfl)
        assert np.array_equal(g.read_value(), ref)


def raw(hj, g, torch):
    out = torch.empty(tuple(g.info().n), device="cuda",
                      dtype={hj.HJ_FP64: torch.float64, hj.HJ_FP32: torch.float32, hj.HJ_Q527: torch.int32}[g.info().precision])
    return g.read_value_device(out).cpu().numpy()


@pytest.mark.parametrize("prec, kernel", [("FP64", "GENERIC"), ("FP32", "GENERIC"), ("FP32", "TILED"),
                                          ("Q527", "TILED"), ("Q527", "GENERIC"), ("FP32", "RESIDENT"),
                                          ("FP64", "RESIDENT"), ("Q527", "RESIDENT")])
@pytest.mark.parametrize("first", [0, 3])
def test_failed_launch_keeps_value_and_step_count_together(hj, prec, kernel, first):
    """The launch of step `first` + 6 fails: six steps less one were queued
    before it (none with the resident kernel, whose launch is a whole call)."""
    import torch
    w = scenes.workload("car4d_31x31x11x16")
    V0 = scenes.initial_value(w.grid, w.scene)
    ran = 0 if kernel == "RESIDENT" else 5
    with hj.Grid.for_workload(w, getattr(hj, "HJ_" + prec)) as g:
        g.set_kernel(getattr(hj, "HJ_KERNEL_" + kernel))
        g.set_initial_value(V0)
        st = g.advance_brt(w.T, w.cfl, first + ran)
        after, t_after = raw(hj, g, torch), st.t_final
        g.solve_brt(w.T, w.cfl)
        end = raw(hj, g, torch)
        for call in (lambda: g.solve_brt(w.T, w.cfl), lambda: g.solve_converged(1e-9, w.T, w.cfl)):
            g.set_initial_value(V0)
            if first:
                g.advance_brt(w.T, w.cfl, first)
            hj.hj_launch_selftest(g.handle, ran + 1)
            with pytest.raises(hj.HjError) as e:
                call()
            assert e.value.status == hj.HJ_ERR_CUDA
            info = g.info()
            assert info.has_value and info.total_steps == first + ran and info.t == t_after
            assert np.array_equal(raw(hj, g, torch), after)
            st = g.solve_brt(w.T, w.cfl)
            assert np.array_equal(raw(hj, g, torch), end)


def test_failed_autotune_leaves_the_grid_ready(hj):
    w = scenes.workload("car4d_31x31x11x16")
    V0 = scenes.initial_value(w.grid, w.scene)
    with hj.Grid.for_workload(w, hj.HJ_FP32) as g:
        g.set_kernel(hj.HJ_KERNEL_TILED)
        g.set_initial_value(V0)
        tile = list(g.info().tile)
        hj.hj_launch_selftest(g.handle, 3)
        with pytest.raises(hj.HjError):
            g.autotune(4)
        assert list(g.info().tile) == tile and g.info().total_steps == 0
        g.solve_brt(w.T, w.cfl)
        V = g.read_value()
    with hj.Grid.for_workload(w, hj.HJ_FP32) as g:
        g.set_kernel(hj.HJ_KERNEL_TILED)
        g.set_initial_value(V0)
        g.solve_brt(w.T, w.cfl)
        assert np.array_equal(g.read_value(), V)


@pytest.mark.parametrize("prec", ["FP32", "Q527"])
@pytest.mark.parametrize("xy", [False, True])
@pytest.mark.parametrize("threshold", [0.0, 1e-3])
@pytest.mark.parametrize("n", [(31, 31, 11, 16), (12, 10, 9, 33)])
def test_steps_behind_a_timed_out_one_leave_at_once(hj, prec, xy, threshold, n):
    w = scenes.custom_workload(n, n_circles=3, T=0.4, seed=sum(n))
    V0 = scenes.initial_value(w.grid, w.scene)
    out = []
    with hj.Grid.for_workload(w, getattr(hj, "HJ_" + prec)) as g:
        g.set_kernel(hj.HJ_KERNEL_TILED)
        for _ in range(2):
            if xy:
                g.set_initial_value_xy(scenes.signed_distance_xy(w.grid, w.scene))
            else:
                g.set_initial_value(V0)
            if not out:
                assert hj.hj_stop_selftest(g.handle, w.T, w.cfl, threshold) == (hj.HJ_ERR_TIMEOUT, 0)
                # the value is gone and the status stays until the next V0
                assert not g.info().has_value
                with pytest.raises(hj.HjError) as e:
                    g.read_value()
                assert e.value.status == hj.HJ_ERR_STATE
                with pytest.raises(hj.HjError) as e:
                    g.solve_brt(w.T, w.cfl)
                assert e.value.status == hj.HJ_ERR_TIMEOUT
                if xy:
                    g.set_initial_value_xy(scenes.signed_distance_xy(w.grid, w.scene))
                else:
                    g.set_initial_value(V0)
            g.solve_brt(w.T, w.cfl)
            out.append(g.read_value())
    assert np.array_equal(out[0], out[1])
    with hj.Grid.for_workload(w, getattr(hj, "HJ_" + prec)) as g:
        g.set_kernel(hj.HJ_KERNEL_TILED)
        g.set_initial_value(V0)
        g.solve_brt(w.T, w.cfl)
        assert np.array_equal(g.read_value(), out[0])


@pytest.mark.parametrize("launch", [1, 7, 60])
def test_failed_autotune_at_any_trial_leaves_status_and_steps(hj, launch):
    """A launch that fails in the first trial, in a later one, and (if there are
    so many) among the re-timed shapes: the grid then solves as a new one."""
    w = scenes.custom_workload((40, 41, 16, 24), n_circles=3, T=0.3, seed=11)
    V0 = scenes.initial_value(w.grid, w.scene)
    out = []
    for tuned in (False, True):
        with hj.Grid.for_workload(w, hj.HJ_FP32) as g:
            g.set_kernel(hj.HJ_KERNEL_TILED)
            g.set_initial_value(V0)
            if tuned:
                hj.hj_launch_selftest(g.handle, launch)
                try:
                    g.autotune(2)
                except hj.HjError as e:
                    assert e.status == hj.HJ_ERR_CUDA
                hj.hj_launch_selftest(g.handle, 0)
            st = g.solve_brt(w.T, w.cfl)
            out.append((g.read_value(), st.steps, st.t_final))
    assert out[0][1:] == out[1][1:] and np.array_equal(out[0][0], out[1][0])
