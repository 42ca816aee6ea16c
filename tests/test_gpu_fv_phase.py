"""The two-launch FV step (LB_FV_TILE, chunk 2; the default on FP64 and small
grids) element by element against the FP64 oracle, on both of its forms and
at the sizes where they change: one population per thread at 8 and at 32
cells per CTA, one cell per thread on larger FP64 grids; periodic and wall
axes, ragged last CTAs, axes shorter than the stencil."""
import numpy as np
import pytest

from tests import inputs
from tests.test_gpu_parity import pair

pytestmark = pytest.mark.gpu

CASES = [
    dict(nx=1, ny=64, lx=1.0),
    dict(nx=3, ny=2, bcy=1),
    dict(nx=2, ny=5, bcx=1),
    dict(nx=35, ny=34, sx=1, stretch_x=1.0, sy=2, stretch_y=4.0, bcx=1, bcy=1),
    dict(nx=33, ny=41, sy=1, stretch_y=2.0, bcy=1, thermal=True),
    dict(nx=9, ny=7, thermal=True),
    # past the eight cells per SM, and past the sizes by population (FP64)
    dict(nx=61, ny=45, bcx=1),
    dict(nx=64, ny=38, sy=1, stretch_y=2.0, bcy=1, thermal=True),
    dict(nx=151, ny=109, sx=3, bcx=1, bcy=1),
    dict(nx=151, ny=109, bcx=1),
    dict(nx=150, ny=109, sy=1, stretch_y=1.5, bcy=1),
    dict(nx=151, ny=109),
    dict(nx=101, ny=82, sy=1, stretch_y=2.0, bcy=1, thermal=True),
    dict(nx=101, ny=82, thermal=True),
]


@pytest.mark.parametrize("store", ["f64", "f32"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(f"{k}{v}" for k, v in c.items()))
def test_two_launch_step(lbgpu, oracle, case, store):
    """After 3 steps every population agrees to 1e-13 (FP64), or to 2e-6 of
    the deviation scale (FP32), the bars of the other schedules."""
    nx, ny, th = case["nx"], case["ny"], case.get("thermal", False)
    kw = dict(tau=0.3, dt=0.05, ax=2e-4, ay=-1e-4)
    if th:
        kw.update(tau_g=0.25, beta=1e-2, grav=1.0, T0=1.0, T_bot=1.3, T_top=0.8)
    g, r = pair(lbgpu, oracle, store=lbgpu.STORE_NAMES[store], **case, **kw)
    g.set_fv_schedule(lbgpu.LB_FV_TILE, 2)
    assert g.fv_schedule() == (lbgpu.LB_FV_TILE, 2)
    g.set_pops(inputs.random_populations(nx, ny, seed=3 * nx + ny, amp=0.2),
               inputs.random_populations(nx, ny, seed=11, amp=0.2) if th else None)
    start = g.get_pops()  # both sides from the stored state
    r.set_pops(*start)
    g.step_fv(2)  # h is formed again at each call
    g.step_fv(1)
    r.step_fv(3)
    wts = oracle.lattice()[2][:, None, None]
    for a, b, s, T0 in zip(g.get_pops(), r.get_pops(), start, (1.0, kw.get("T0"))):
        if s is not None:
            tol = 1e-13 if store == "f64" else 2e-6 * np.abs(s - wts * T0).max()
            assert np.abs(a - b).max() <= tol


@pytest.mark.parametrize("store", ["f16dev", "bf16dev"])
def test_two_launch_step_16bit(lbgpu, store):
    """16-bit storage: the two launches and the paired tile round the same
    states, so after one step they differ by at most one rounding of the
    stored deviations (2^-10 and 2^-7 of the largest)."""
    out = []
    for sched in ((4, 0), (1, 2)):
        g = lbgpu.Grid(40, 36, sy=1, stretch_y=2.0, bcy=1, thermal=True, store=store)
        g.init(tau=0.1, tau_g=0.1, dt=0.05, beta=1e-3, grav=1.0, T0=1.0, T_bot=1.5, T_top=0.5, kind=lbgpu.LB_INIT_RB,
               amp=1e-2, seed=5)
        g.set_pops(inputs.random_populations(40, 36, seed=2, amp=0.1), inputs.random_populations(40, 36, seed=3, amp=0.1))
        out.append(g.set_fv_schedule(*sched).step_fv(1).get_pops())
    ulp = 2.0 ** -10 if store == "f16dev" else 2.0 ** -7
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= ulp * max(np.abs(a - w).max(), 0.05)


@pytest.mark.parametrize("nx,ny,thermal,store,two", [
    (64, 64, False, "f32", True), (1024, 8, False, "f64", True), (200, 200, False, "f32", False),
    (64, 64, True, "f16dev", True), (128, 128, True, "f32", False)])
def test_default_schedule(lbgpu, nx, ny, thermal, store, two):
    """FP64 grids and small FP32-math ones take the two launches, counted as
    one launch for h and two per step; replays of a graph change no bit."""
    outs = []
    for n in (0, 8):
        g = lbgpu.Grid(nx, ny, bcy=1, thermal=thermal, store=store)
        assert (g.fv_schedule() == (lbgpu.LB_FV_TILE, 2)) == two
        g.init(tau=0.3, dt=0.2, kind=lbgpu.LB_INIT_TGV, u0=0.02).set_graph_steps(n)
        l0 = lbgpu.lb_kernel_launches()
        g.step_fv(21)
        assert lbgpu.lb_kernel_launches() - l0 == (43 if two else 21)
        outs.append(g.get_pops()[0])
    assert np.array_equal(outs[0], outs[1])
