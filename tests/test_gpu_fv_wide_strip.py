"""The block march's wide flow strip (120 columns, one CTA per SM), which its
step costs choose from about 480 columns, and every shape of the paired tile:
one step, bit for bit, on grids whose last strip has 1, 3, 41 and 9 columns,
with ragged and whole blocks of rows, periodic and walled.  And served requests
of those sizes against a grid stepped on the paired tile, exactly."""
import numpy as np
import pytest

from tests import inputs

pytestmark = pytest.mark.gpu

KW = dict(tau=0.3, dt=0.05, ax=2e-4, ay=-1e-4)
TH = dict(KW, tau_g=0.25, beta=1e-2, grav=1.0, T0=1.0, T_bot=1.3, T_top=0.8)
WALLS = dict(sy=1, stretch_y=2.0, bcy=1)


def _compare(lb, nx, ny, thermal, store, geo, scheds):
    grid = lb.Grid(nx, ny, thermal=thermal, store=store, **geo).init(**(TH if thermal else KW))
    f = inputs.random_populations(nx, ny, seed=nx, amp=0.2)
    g = inputs.random_populations(nx, ny, seed=ny, amp=0.2) if thermal else None
    want = None
    for s in scheds:
        out = grid.set_pops(f, g).set_fv_schedule(*s).step_fv(3).get_pops()
        if want is None:
            want = out
        assert np.array_equal(out[0], want[0]), s
        assert not thermal or np.array_equal(out[1], want[1]), s
    grid.close()


# chunks for which the step costs choose the wide strip on 152 SMs
WIDE = [(1001, 335, (0, 4, 8, 32)), (1089, 641, (0, 4, 16, 64)), (483, 301, (0, 8, 16)), (241, 1030, (8, 16, 32))]
TILES = ((4, 0), (4, 14), (4, 16), (4, 512), (4, 526))


@pytest.mark.parametrize("geo", [{}, WALLS], ids=["periodic", "walls"])
@pytest.mark.parametrize("nx,ny,chunks", WIDE)
def test_wide_strip_is_the_tile(lbgpu, nx, ny, chunks, geo):
    _compare(lbgpu, nx, ny, False, "f32", geo, TILES + tuple((3, c) for c in chunks) + ((3, 128),))


@pytest.mark.parametrize("store", ["f16dev", "bf16dev"])
def test_wide_strip_in_16_bits(lbgpu, store):
    _compare(lbgpu, 1001, 335, False, store, WALLS, TILES + ((3, 0), (3, 32)))


@pytest.mark.parametrize("store", ["f32", "f16dev", "bf16dev"])
def test_thermal_strip_is_the_tile(lbgpu, store):
    _compare(lbgpu, 617, 333, True, store, WALLS, TILES + ((3, 0), (3, 8), (3, 64)))


RB = dict(TH, tau=0.05, tau_g=0.05, beta=2e-4, T_bot=1.5, T_top=0.5, dt=0.1, amp=1e-2, ax=0.0, ay=0.0)
FLOW = dict(tau=0.1, dt=0.5, u0=0.01)


def _serve(lb, reqs, store, thermal):
    s = lb.Server(store=store, thermal=thermal, steps_per_launch=8)
    n0 = lb.lb_kernel_launches()
    for i, (nx, ny) in enumerate(reqs):
        s.submit(i, 16, nx, ny, seed=i + 1, kind=lb.LB_INIT_RB if thermal else lb.LB_INIT_TGV,
                 **(dict(WALLS, **RB) if thermal else FLOW))
    out = {}
    while len(out) < len(reqs):
        s.pump()
        out.update({r["id"]: r for r in s.results()})
    s.close()
    return out, lb.lb_kernel_launches() - n0


@pytest.mark.parametrize("store,thermal", [("f16dev", True), ("f32", True), ("f32", False), ("bf16dev", False)])
def test_served_figures_are_the_tiles(lbgpu, store, thermal):
    """A second large request adds 16 launches of its own for its 16 steps, a
    second small one none; the figures equal the paired tile's."""
    lb = lbgpu
    big, small = [(1001, 635), (1089, 641)], [(64, 40), (96, 64)]
    out, n2 = _serve(lb, big, store, thermal)
    _, n1 = _serve(lb, big[:1], store, thermal)
    _, m2 = _serve(lb, small, store, thermal)
    _, m1 = _serve(lb, small[:1], store, thermal)
    assert (n2 - n1) - (m2 - m1) == 16
    for i, (nx, ny) in enumerate(big):
        g = lb.Grid(nx, ny, thermal=thermal, store=store, **(WALLS if thermal else {}))
        g.init(kind=lb.LB_INIT_RB if thermal else lb.LB_INIT_TGV, seed=i + 1, **(RB if thermal else FLOW))
        g.set_fv_schedule(lb.LB_FV_PTILE).step_fv(16)
        assert out[i]["mass"] == g.conservation()[0]
        if thermal:
            assert (out[i]["nu_vol"], out[i]["nu_bot"], out[i]["nu_top"]) == tuple(g.nusselt())
        g.close()
