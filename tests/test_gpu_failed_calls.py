"""Calls that fail leave a grid as it was, or say that its value is gone: a
call on a stream that is being captured."""
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
