"""The two-launch FV step (LB_FV_TILE, chunk 2; the default on FP64 and small
grids) element by element against the FP64 oracle, on both of its forms and
at the sizes where they change: one population per thread at 8 and at 32
cells per CTA, one cell per thread on larger FP64 grids; periodic and wall
axes, ragged last CTAs, axes shorter than the stencil.  And the packed FP32
schedules (tile, block march, two launches) against each other, bit for bit."""
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


PAIRED = [  # x-periodic grids: ragged tiles and blocks, walls in every position of a block, axes shorter than a stencil
    dict(nx=70, ny=37), dict(nx=45, ny=33, sy=1, stretch_y=2.0, bcy=1), dict(nx=5, ny=3), dict(nx=64, ny=2, bcy=1),
    dict(nx=1, ny=9), dict(nx=33, ny=4, bcy=1), dict(nx=40, ny=5, sy=1, stretch_y=2.0, bcy=1), dict(nx=61, ny=6, bcy=1),
    dict(nx=50, ny=7, sy=1, stretch_y=2.0, bcy=1), dict(nx=250, ny=66, sy=1, stretch_y=2.0, bcy=1)]


@pytest.mark.parametrize("store", ["f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("thermal", [False, True], ids=["flow", "thermal"])
@pytest.mark.parametrize("case", PAIRED, ids=lambda c: "-".join(f"{k}{v}" for k, v in c.items()))
def test_packed_schedules_are_one_step(lbgpu, case, thermal, store):
    """The paired tile, the block march (chunks of one block, of several, of
    the whole grid, the automatic one) and the two-launch step form the same
    values in the same order: equal populations, bit for bit."""
    kw = dict(tau=0.3, dt=0.05, ax=2e-4, ay=-1e-4)
    if thermal:
        kw.update(tau_g=0.25, beta=1e-2, grav=1.0, T0=1.0, T_bot=1.3, T_top=0.8)
    nx, ny, out = case["nx"], case["ny"], []
    grid = lbgpu.Grid(**case, thermal=thermal, store=store).init(**kw)
    f = inputs.random_populations(nx, ny, seed=1, amp=0.2)
    g = inputs.random_populations(nx, ny, seed=2, amp=0.2) if thermal else None
    for sched in ((4, 0), (4, 526), (4, 16), (3, 4), (3, 8), (3, 12), (3, 64), (3, 0), (1, 2)):
        out.append(grid.set_pops(f, g).set_fv_schedule(*sched).step_fv(3).get_pops())
    for o in out[1:]:
        assert np.array_equal(o[0], out[0][0])
        assert not thermal or np.array_equal(o[1], out[0][1])


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
