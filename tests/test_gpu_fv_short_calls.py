"""Calls of a few FV steps: the two-launch step pays a third launch per call,
so on FP32-math grids the default leaves such calls to the paired tile, whose
bits are the same; FP64 grids keep the two launches at every length."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KW = dict(tau=0.3, dt=0.05, ax=2e-4, ay=-1e-4, u0=0.02)
TH = dict(KW, tau_g=0.25, beta=1e-2, grav=1.0, T0=1.0, T_bot=1.3, T_top=0.8, amp=0.01)


def _launches(lb, g, n):
    l0 = lb.lb_kernel_launches()
    g.step_fv(n)
    return lb.lb_kernel_launches() - l0


@pytest.mark.parametrize("nx,ny,thermal,store,one,long", [
    (64, 64, False, "f32", 1, 43), (16, 16, False, "bf16dev", 1, 43), (120, 120, False, "f32", 1, 43),
    (98, 98, True, "f16dev", 1, 43), (40, 40, True, "f32", 1, 43), (64, 64, False, "f64", 3, 43)])
def test_one_step_calls(lbgpu, nx, ny, thermal, store, one, long):
    lb = lbgpu
    g = lb.Grid(nx, ny, bcy=1, thermal=thermal, store=store)
    outs = []
    for calls in ([1] * 21, [21], [2, 3, 16]):
        g.init(kind=lb.LB_INIT_TGV, **(TH if thermal else KW))
        n = [_launches(lb, g, k) for k in calls]
        assert n == ([one] * 21 if len(calls) == 21 else [long] if len(calls) == 1 else n)
        outs.append(g.get_pops())
    for o in outs[1:]:
        assert np.array_equal(o[0], outs[0][0])
        assert not thermal or np.array_equal(o[1], outs[0][1])
    # asked for, the two launches run at every length
    assert _launches(lb, g.set_fv_schedule(lb.LB_FV_TILE, 2), 1) == 3


def test_autotune_times_whole_calls(lbgpu):
    """Tuned for calls of one step, a 64 x 64 FP32 grid (three launches, 6.3 us,
    against the paired tile's 5.2) does not take the two launches; tuned for long ones it does."""
    lb = lbgpu
    g = lb.Grid(64, 64, store="f32").init(kind=lb.LB_INIT_TGV, **KW)
    assert g.autotune_fv(1) != (lb.LB_FV_TILE, 2)
    assert g.autotune_fv(200) == (lb.LB_FV_TILE, 2)
