"""Which passes a 3-D FV call takes, by its launches: the default on small FP32
grids is two passes a step after one that forms h (1 + 2 n), the staged
passes are four (4 n); and the autotuner does not lose the two passes."""
import numpy as np
import pytest

from tests.test_gpu_3d import STAGED_CASES, _ids, _params

pytestmark = pytest.mark.gpu


def _launches(lb, g, n):
    l0 = lb.lb_kernel_launches()
    g.step_fv(n)
    return lb.lb_kernel_launches() - l0


@pytest.mark.parametrize("case", STAGED_CASES + [dict(nx=128, ny=9, nz=7, bcz=1, thermal=True)], ids=_ids)
def test_small_grids_take_two_passes(lbgpu, case):
    lb = lbgpu
    g = lb.Grid3(**case, store=lb.LB_STORE_F32).init(**_params(case.get("thermal", False)))
    assert [_launches(lb, g, n) for n in (1, 3)] == [3, 7]
    g.set_fv_schedule(lb.LB3_FV_STAGED)
    assert [_launches(lb, g, n) for n in (1, 3)] == [4, 12]
    g.close()


def test_autotune_keeps_two_passes(lbgpu):
    """Thermal 32 x 40 x 20, 20 steps: two passes 27 us a step, four staged ones 43."""
    lb = lbgpu
    geo = dict(lz=20.0, sz=lb.LB_AXIS_TANH, stretch_z=1.5, bcz=lb.LB_BC_WALLS, thermal=True)
    kw = dict(tau=0.2, tau_g=0.2, dt=0.2, beta=1e-2, grav=1.0, T0=1.0, T_bot=1.5, T_top=0.5)
    outs = []
    for tune in (False, True):
        g = lb.Grid3(32, 40, 20, **geo).init(**kw, kind=lb.LB_INIT_RB, amp=1e-2, seed=11)
        if tune:
            g.autotune_fv(20)
        assert _launches(lb, g, 5) == 11
        outs.append(g.get_pops())
        g.close()
    for a, b in zip(*outs):
        assert np.array_equal(a, b)


def test_one_step_calls_of_larger_thermal_grids(lbgpu):
    """Thermal 64 x 64 x 32: one step in four passes, more in two each, with the
    bits of one call."""
    lb = lbgpu
    kw = dict(tau=0.2, tau_g=0.2, dt=0.2, beta=1e-2, grav=1.0, T0=1.0, T_bot=1.5, T_top=0.5)
    outs = []
    for calls, launches in (([1, 1, 2], [4, 4, 5]), ([4], [9])):
        g = lb.Grid3(64, 64, 32, bcz=1, thermal=True).init(**kw, kind=lb.LB_INIT_RB, amp=1e-2, seed=11)
        assert [_launches(lb, g, n) for n in calls] == launches
        outs.append(g.get_pops())
        g.close()
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
