"""A run of FV steps has the same bits however it is split into calls: the
two-launch step forms h of a call's first state in a kernel of its own, with
the roundings of the steps before it.  Both FP64 forms (one population and
one cell per thread), with forces, walls and temperature, and 16-bit storage."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KW = dict(tau=0.3, dt=0.05, ax=2e-4, ay=-1e-4, u0=0.02)
TH = dict(KW, tau_g=0.25, beta=1e-2, grav=1.0, T0=1.0, T_bot=1.3, T_top=0.8, amp=0.01)


@pytest.mark.parametrize("store", ["f64", "f32", "f16dev"])
@pytest.mark.parametrize("thermal", [False, True], ids=["flow", "thermal"])
@pytest.mark.parametrize("nx,ny", [(20, 20), (70, 61), (160, 140)])
def test_split_calls_are_one_run(lbgpu, nx, ny, thermal, store):
    g = lbgpu.Grid(nx, ny, sy=1, stretch_y=2.0, bcy=1, thermal=thermal, store=store)
    outs = []
    for calls in ([24], [1] * 24, [5, 7, 12]):
        g.init(kind=lbgpu.LB_INIT_TGV, **(TH if thermal else KW)).set_fv_schedule(lbgpu.LB_FV_TILE, 2)
        for n in calls:
            g.step_fv(n)
        outs.append(g.get_pops())
    g.close()
    for o in outs[1:]:
        assert np.array_equal(o[0], outs[0][0])
        assert not thermal or np.array_equal(o[1], outs[0][1])
