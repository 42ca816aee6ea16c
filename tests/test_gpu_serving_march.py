"""Served requests large enough for the block march: alone, in a mix, and on
either side of the size where they leave the batched tiles, with the figures
of a grid that steps on the paired tile."""
import pytest

pytestmark = pytest.mark.gpu

RB = dict(tau=0.05, tau_g=0.05, beta=2e-4, grav=1.0, T0=1.0, T_bot=1.5, T_top=0.5, dt=0.1, amp=1e-2)
PLATES = dict(sy=1, stretch_y=2.0, bcy=1)


def _serve(lb, reqs, store, thermal, k, policy=0):
    s = lb.Server(store=store, thermal=thermal, steps_per_launch=k, policy=policy)
    for i, (nx, ny, n) in enumerate(reqs):
        s.submit(i, n, nx, ny, seed=i + 1, kind=lb.LB_INIT_RB if thermal else lb.LB_INIT_TGV, **_case(thermal))
    out = {}
    while len(out) < len(reqs):
        s.pump()
        out.update({r["id"]: r for r in s.results()})
    s.close()
    return out


def _case(thermal):
    return {**PLATES, **RB} if thermal else dict(tau=0.1, dt=0.5, u0=0.01)


@pytest.mark.parametrize("store, thermal", [("f16dev", True), ("bf16dev", True), ("f32", True), ("f32", False)])
@pytest.mark.parametrize("k", [7, 70])  # plain launches; a captured graph and a remainder
def test_large_requests_take_the_march(lbgpu, store, thermal, k):
    lb = lbgpu
    reqs = [(601, 607, 23), (64, 40, 30), (1024, 333, 9), (1088, 640, 75)]
    mix = _serve(lb, reqs, store, thermal, k)
    tol = 1e-7 if store == "f32" else 1e-5  # plate Nu amplifies rounding by ~H * 20
    for i, (nx, ny, n) in enumerate(reqs):
        r = mix[i]
        assert r["status"] == lb.LB_OK and r["steps"] == n
        g = lb.Grid(nx, ny, thermal=thermal, store=store, **(PLATES if thermal else {}))
        kw = RB if thermal else _case(False)
        g.init(kind=lb.LB_INIT_RB if thermal else lb.LB_INIT_TGV, seed=i + 1, **kw)
        g.set_fv_schedule(lb.LB_FV_PTILE)
        g.step_fv(n)
        want = [g.conservation()[0]] + (list(g.nusselt()) if thermal else [])
        got = [r["mass"]] + ([r["nu_vol"], r["nu_bot"], r["nu_top"]] if thermal else [])
        g.close()
        for a, b in zip(got, want):
            assert abs(a - b) <= tol * abs(b)


@pytest.mark.parametrize("policy", [0, 1, 2], ids=["share", "shortest", "arrival"])
def test_alone_equals_mix_large(lbgpu, policy):
    """One large request (no tiles in the table at all) and the same one among others."""
    reqs = [(700, 640, 20), (96, 64, 31), (640, 704, 13)]
    mix = _serve(lbgpu, reqs, "f16dev", True, 8, policy)
    one = _serve(lbgpu, reqs[:1], "f16dev", True, 8)
    for key in ("status", "steps", "mass", "nu_vol", "nu_bot", "nu_top"):
        assert one[0][key] == mix[0][key]
