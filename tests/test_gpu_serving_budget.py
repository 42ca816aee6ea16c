"""The server reserves what a grid allocates: on narrow grids the per-row
tables (about 230 bytes a row) count, not a fixed 64 bytes."""
import pytest

pytestmark = pytest.mark.gpu

RB = dict(tau=0.05, tau_g=0.05, beta=2e-4, grav=1.0, T0=1.0, T_bot=1.5, T_top=0.5, dt=0.1, amp=1e-3)


def test_reservation_counts_the_tables(lbgpu):
    lb, nx, ny = lbgpu, 4, 20000
    state = 2 * 2 * 9 * 32 * 4 * ny + 4 * 8 * nx * ny  # f and g twice at a pitch of 32, staging fields

    def server(per_row):
        return lb.Server(store="f32", thermal=True, hbm_budget=state + per_row * ny + 65536, steps_per_launch=2)

    s = server(200)
    with pytest.raises(lb.LBError) as e:
        s.submit(rid=1, nsteps=2, nx=nx, ny=ny, bcy=1, **RB)
    assert e.value.status == lb.LB_ERR_ARG
    s.close()
    s = server(260)
    s.submit(rid=1, nsteps=2, nx=nx, ny=ny, bcy=1, **RB)
    s.submit(rid=2, nsteps=2, nx=nx, ny=0, bcy=1, **RB)  # an invalid size fails by itself, in the pump
    got = {}
    while len(got) < 2:
        s.pump()
        got.update({r["id"]: r for r in s.results()})
    s.close()
    assert got[1]["status"] == lb.LB_OK and got[2]["status"] == lb.LB_ERR_ARG
