"""lb_get_fv_schedule names the tile that a step runs: 32 x 16 where the two
launches were asked for on a grid they do not serve, and on grids with a
density axis or a single-stage scheme, which AUTO gives no smaller tile."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw,scheme", [
    (dict(bcx=2), 0), (dict(bcx=1, bcy=2), 0), (dict(bcx=1, bcy=1), 2), (dict(bcx=1), 1)])
@pytest.mark.parametrize("asked", [(1, 2), (0, 0)])
def test_scalar_tile_reported(lbgpu, kw, scheme, asked):
    lb = lbgpu
    g = lb.Grid(40, 30, store="f32", **kw).set_fv_scheme(scheme).set_fv_schedule(*asked)
    assert g.fv_schedule() == (lb.LB_FV_TILE, 0)
    g.init(tau=0.3, dt=0.1, kind=lb.LB_INIT_TGV, u0=0.01)
    n0 = lb.lb_kernel_launches()
    g.step_fv(3)
    assert lb.lb_kernel_launches() - n0 == 3
    g.close()
