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


def test_chunk_of_the_march_stays_positive(lbgpu):
    """Any chunk beyond the grid is the whole grid."""
    g = lbgpu.Grid(64, 40, store="f32")
    for chunk in (2**31 - 1, 2**31 - 8, 4096):
        g.set_fv_schedule(lbgpu.LB_FV_PAIR, chunk)
        assert 40 <= g.fv_schedule()[1] <= chunk
        g.init(tau=0.3, dt=0.1, kind=lbgpu.LB_INIT_TGV, u0=0.01).step_fv(2).sync()
    g.close()
