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


@pytest.mark.parametrize("nx,ny,shape", [(100, 100, 8), (333, 257, 16), (420, 270, 0), (460, 300, 0), (470, 330, 16),
                                         (470, 500, 16), (470, 600, 0), (300, 1200, 16)])
def test_default_tile_between_x_walls(lbgpu, nx, ny, shape):
    """The tile that is fastest at each size (csrc/lb_abi.cu, scalar_shape; on
    152 SMs), with the populations of the 32 x 16 tile to FP32 rounding."""
    import numpy as np
    lb = lbgpu
    g = lb.Grid(nx, ny, bcx=1, bcy=1, store="f32")
    outs = []
    for sched in ((0, 0), (1, 0)):
        g.init(tau=0.3, dt=0.05, kind=lb.LB_INIT_TGV, u0=0.02).set_fv_schedule(*sched)
        assert g.fv_schedule() == (lb.LB_FV_TILE, 0 if sched[0] else shape)
        outs.append(g.step_fv(3).get_pops()[0])
    wts = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    assert np.abs(outs[0] - outs[1]).max() <= 2e-6 * np.abs(outs[1] - wts).max()
    g.close()
