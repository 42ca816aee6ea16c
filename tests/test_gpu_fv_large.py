"""Grids whose planes reach 32-bit limits: the schedules that address planes
with 32-bit offsets give the bits of those that use 64 bits throughout."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RB = dict(tau=0.3, tau_g=0.25, beta=2e-4, grav=1.0, T0=1.0, T_bot=1.5, T_top=0.5, dt=0.05, amp=1e-2, seed=5)


def _need(gib):
    import torch
    if torch.cuda.mem_get_info()[0] < gib << 30:
        pytest.skip(f"needs {gib} GiB of free device memory")


def test_two_launches_past_2_32_elements(lbgpu):
    """18 planes of 2^28 cells are 2^32 elements and more: plane 16 of the
    two-launch step's fields is not plane 0.  Windows at the first and the
    last rows, where every population is far from every other's plane."""
    _need(100)
    lb, n = lbgpu, 16384
    wins = []
    with_two = ((lb.LB_FV_PTILE, 0), (lb.LB_FV_TILE, 2))
    g = lb.Grid(n, n, bcy=lb.LB_BC_WALLS, thermal=True, store="bf16dev")
    try:
        for sched in with_two:
            g.init(kind=lb.LB_INIT_RB, **RB).set_fv_schedule(*sched)
            assert g.fv_schedule() == sched
            n0 = lb.lb_kernel_launches()
            g.step_fv(2)
            assert lb.lb_kernel_launches() - n0 == (5 if sched[0] == lb.LB_FV_TILE else 2)
            wins.append([g.get_window(x, y, 64, 48) for x, y in ((0, 0), (n - 32, n // 2), (n // 3, n - 48))])
    finally:
        g.close()
    for a, b in zip(*wins):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
