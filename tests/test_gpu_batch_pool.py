"""Memory of removed slots that a batch keeps for the next ones: it is given
up when another allocation of the library needs it, and it follows the sizes
that are served."""
import numpy as np
import pytest

from paper_2012_04011_gb300 import scenes

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def hj():
    from paper_2012_04011_gb300 import _build
    _build.build()
    from paper_2012_04011_gb300 import hj as mod
    return mod


def add_and_remove(b, n):
    b.remove(b.add_workload(scenes.custom_workload(n, n_circles=1, T=0.1, seed=1)))


def test_kept_memory_is_given_up_to_a_grid(hj):
    import torch
    w = scenes.custom_workload((64, 64, 64, 64), n_circles=3, T=0.05, seed=2)  # 192 MB of values
    small = scenes.workload("car4d_31x31x11x16")
    with hj.Grid.for_workload(small, hj.HJ_FP32) as g:  # (kernels loaded before the device is filled)
        g.set_initial_value(scenes.initial_value(small.grid, small.scene))
        g.solve_brt(small.T, small.cfl)
    with hj.Grid.for_workload(w, hj.HJ_FP32) as g:
        g.set_initial_value(scenes.initial_value(w.grid, w.scene))
        g.solve_brt(w.T, w.cfl)
        ref = g.read_value()
    with hj.Batch(4, memory_budget=1 << 31) as b:
        for n in ((100, 100, 30, 80), (100, 100, 30, 84)):  # 275 and 288 MB, kept
            add_and_remove(b, n)
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        fill = torch.empty(free - 150 * MB, dtype=torch.uint8, device="cuda")
        try:
            with hj.Grid.for_workload(w, hj.HJ_FP32) as g:
                g.set_initial_value(scenes.initial_value(w.grid, w.scene))
                g.solve_brt(w.T, w.cfl)
                assert np.array_equal(g.read_value(), ref)
            # and what does not fit even so is still refused
            with pytest.raises(hj.HjError) as e:
                hj.Grid((128, 128, 64, 96), scenes.DOMAIN_LO, scenes.DOMAIN_HI, scenes.PERIODIC_THETA, hj.HJ_FP32)
            assert e.value.status == hj.HJ_ERR_OOM
        finally:
            del fill
            torch.cuda.empty_cache()
        add_and_remove(b, (100, 100, 30, 80))


def test_kept_memory_follows_the_sizes_that_are_served(hj):
    import torch
    old, new = (128, 128, 44, 96), (100, 100, 48, 84)  # 794 and 461 MB: both are more than is kept
    with hj.Batch(2, memory_budget=1 << 32) as b:
        free = lambda: torch.cuda.mem_get_info()[0]  # noqa: E731
        add_and_remove(b, old)
        for _ in range(70):  # the first size is not asked for again
            add_and_remove(b, new)
        before = free()
        slot = b.add_workload(scenes.custom_workload(new, n_circles=1, T=0.1, seed=1))
        assert before - free() < 64 * MB  # a block of that size was there
        b.remove(slot)
        # never more than 1 GiB is kept
        for k in range(4):
            add_and_remove(b, (100, 100, 48, 80 - 4 * k))
        kept = -free()
    kept += free()
    assert 0 <= kept <= 1024 * MB + 128 * MB
