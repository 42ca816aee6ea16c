"""The work this library is used for, as cases that can be timed and checked.

A pass advances a prepared grid by a number of time steps through the public
entry points and reads the result back into the caller's page-locked arrays:
the macroscopic fields where a run writes snapshots, the populations where it
writes a restart file, the Nusselt numbers and the mass of each request where
it serves a stream.  Grids, parameters and initial states follow
`paper_1505_03271_gb300/configs.py`, `serving.py`, `studies.py`, the benchmark
and the tests.  `exact` computes the same in FP64 with plain torch, written
from the equations of arXiv:1505.03271.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_1505_03271_gb300 as lb

UNIFORM, TANH, SINH, CHEB = lb.LB_AXIS_UNIFORM, lb.LB_AXIS_TANH, lb.LB_AXIS_SINH, lb.LB_AXIS_CHEB
PERIODIC, WALLS = lb.LB_BC_PERIODIC, lb.LB_BC_WALLS


# ------------------------------------------------------------------ cases --

def listed():
    return [
        # Stability and viscosity studies (Figs. KOL, KOL3): a decaying shear
        # wave on a grid one cell wide, FP64, thousands of steps per run; the
        # smallest grids, where a step is a launch.
        _flow("study_wave_1x64_f64", "fv", 1, 64, "f64", 2000, dt=0.5, u=1e-3, out="pops"),
        # The accuracy workload: 64 x 64 decaying vortices in FP64.
        _flow("decay_64x64_f64", "fv", 64, 64, "f64", 1000, dt=0.5, u=0.01, out="pops"),
        # The body-force channel, walls on y refined by tanh, FP32.
        _channel("channel_256x512_f32", 256, 512, "f32", 1000),
        # A closed box with walls on all four sides refined on both axes, odd sizes.
        _flow("box_333x257_f32", "fv", 333, 257, "f32", 500, bc=WALLS, s=TANH, u=0.02, out="pops"),
        # Large periodic flow in FP32 by finite volumes.
        _flow("decay_4096x4096_f32", "fv", 4096, 4096, "f32", 100, dt=0.5, u=0.02, out="fields"),
        # Rayleigh-Benard at Ra = 1e8, 16-bit deviation storage.
        _rb("rb_1024x1024_f16", "fv", 1024, 1024, "f16dev", 400, Ra=1e8, out="pops"),
        # A Rayleigh-Benard layer of aspect ratio 8/3 in FP32, ragged sizes.
        _rb("rb_1000x375_f32", "fv", 1000, 375, "f32", 500, Ra=1e6, out="pops"),
        # Collide-and-stream at the headline size, FP32.
        _flow("stream_8192x8192_f32", "st", 8192, 8192, "f32", 200, dt=1.0, u=0.02, out="fields"),
        # Collide-and-stream with 16-bit deviation storage.
        _flow("stream_4096x4096_f16", "st", 4096, 4096, "f16dev", 400, dt=1.0, u=0.02, out="fields"),
        # The three-dimensional Rayleigh-Benard runs of Table rb, both schemes.
        _rb3("rb3d_fv_128x128x64_f32", "fv", 128, 128, 64, "f32", 100, out="pops"),
        _rb3("rb3d_st_128x128x64_f32", "st", 128, 128, 64, "f32", 300, out="fields"),
        # The serving stream: independent Rayleigh-Benard requests of mixed
        # sizes, Rayleigh numbers and lengths, batched on one GPU.
        {"name": "serve_16_f16", "kind": "serve", "store": "f16dev", "requests": 16, "nmin": 64, "nmax": 512,
         "steps_lo": 50, "steps_hi": 150},
    ]


def draw(rng):
    """One more case of the same ranges."""
    def size(lo, hi):  # log-uniform, any parity
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def steps(cells, per_pass, lo, hi):
        return int(min(hi, max(lo, per_pass / cells)))

    kind = rng.choice(("study", "decay", "channel", "box", "rb", "rb", "stream", "stream16", "rbst", "rb3d", "st3d",
                       "serve"))
    if kind == "study":
        return _flow(None, "fv", rng.choice((1, 2, 3)), size(16, 256), "f64", rng.randint(500, 2000), dt=0.5, u=1e-3,
                     out="pops")
    if kind == "decay":
        nx, ny = size(64, 4096), size(64, 4096)
        store = rng.choice(("f32", "f32", "f16dev", "bf16dev")) if nx * ny > 200 * 200 else rng.choice(("f64", "f32"))
        return _flow(None, "fv", nx, ny, store, steps(nx * ny, 4e8, 60, 500), dt=0.5, u=0.02, out="fields")
    if kind == "channel":
        nx, ny = size(64, 2048), size(64, 1024)
        return _channel(None, nx, ny, rng.choice(("f32", "f32", "f64")), steps(nx * ny, 1e8, 100, 1000))
    if kind == "box":
        nx, ny = size(48, 512), size(48, 512)
        return _flow(None, "fv", nx, ny, rng.choice(("f32", "f64")), steps(nx * ny, 2e7, 100, 500), bc=WALLS, s=TANH,
                     u=0.02, out="pops")
    if kind == "rb":
        nx, ny = size(64, 1536), size(64, 1024)
        return _rb(None, "fv", nx, ny, rng.choice(("f32", "f16dev", "bf16dev")), steps(nx * ny, 2e8, 100, 600),
                   Ra=10.0 ** rng.uniform(4.0, 8.0), out="pops")
    if kind == "rbst":
        nx, ny = size(64, 2048), size(32, 512)
        return _rb(None, "st", nx, ny, rng.choice(("f32", "f64")), steps(nx * ny, 1e8, 100, 1000),
                   Ra=10.0 ** rng.uniform(4.0, 6.0), out="fields")
    if kind in ("stream", "stream16"):
        nx, ny = size(128, 8192), size(128, 8192)
        store = "f32" if kind == "stream" else rng.choice(("f16dev", "bf16dev"))
        return _flow(None, "st", nx, ny, store, steps(nx * ny, 3e9, 100, 1000), dt=1.0, u=0.02, out="fields")
    if kind == "rb3d":
        nx, ny, nz = rng.choice((32, 48, 64, 100, 128, 130, 256)), size(24, 160), 2 * size(10, 48)
        return _rb3(None, "fv", nx, ny, nz, rng.choice(("f32", "f32", "f64")), steps(nx * ny * nz, 3e7, 20, 200),
                    out="pops")
    if kind == "st3d":
        nx, ny, nz = size(24, 192), size(24, 192), size(16, 96)
        return _rb3(None, "st", nx, ny, nz, "f32", steps(nx * ny * nz, 1e8, 50, 400), out="fields")
    return {"kind": "serve", "store": rng.choice(("f16dev", "f32")), "requests": rng.randint(6, 16), "nmin": 48,
            "nmax": size(128, 512), "steps_lo": 30, "steps_hi": rng.randint(60, 150)}


def _named(name, d):
    if name:
        d["name"] = name
    return d


def _flow(name, scheme, nx, ny, store, steps, dt=None, u=0.01, bc=PERIODIC, s=UNIFORM, out="fields"):
    """Decaying vortices of amplitude u, quoted tau = 0.8 (tau = 0.3); without
    dt the step follows the smallest cell."""
    if dt is None:
        dt = 0.5 * min(_widths(nx, float(nx), s, 1.5).min(), _widths(ny, float(ny), s, 1.5).min())
    return _named(name, {"kind": "flow", "scheme": scheme, "nx": nx, "ny": ny, "store": store, "steps": steps,
                         "tau": 0.3, "dt": float(dt), "u": u, "bcx": bc, "bcy": bc, "sx": s, "sy": s,
                         "stretch": 1.5, "ax": 0.0, "out": out})


def _channel(name, nx, ny, store, steps):
    """Walls on y (tanh, delta = 2), quoted tau = 0.7, driven at Re = 10."""
    tau, U = 0.2, 10.0 * (0.2 / 3.0) / ny
    dt = 0.9 * min(_widths(ny, float(ny), TANH, 2.0).min(), 8.0 * tau)
    return _named(name, {"kind": "channel", "scheme": "fv", "nx": nx, "ny": ny, "store": store, "steps": steps,
                         "tau": tau, "dt": float(dt), "u": U, "bcx": PERIODIC, "bcy": WALLS, "sx": UNIFORM,
                         "sy": TANH, "stretch": 2.0, "ax": 8.0 * (tau / 3.0) * U / ny ** 2, "out": "pops"})


def _rb(name, scheme, nx, ny, store, steps, Ra, out):
    """Rayleigh-Benard layer of height ny, free-fall velocity 0.1, Pr = 1."""
    return _named(name, {"kind": "rb", "scheme": scheme, "nx": nx, "ny": ny, "store": store, "steps": steps,
                         "Ra": float(Ra), "bcx": PERIODIC, "bcy": WALLS, "sx": UNIFORM,
                         "sy": TANH if scheme == "fv" else UNIFORM, "stretch": 2.0, "out": out})


def _rb3(name, scheme, nx, ny, nz, store, steps, out):
    """The Table rb parameters on nx x ny x nz cells (plates on z)."""
    return _named(name, {"kind": "rb3", "scheme": scheme, "nx": nx, "ny": ny, "nz": nz, "store": store,
                         "steps": steps, "out": out})


# ------------------------------------------------------- parameters, inputs --

def _faces(n, L, sp, st):
    s = np.arange(n + 1) / n
    if sp == TANH:
        x = 0.5 * L * (1.0 + np.tanh((2.0 * s - 1.0) * st) / math.tanh(st))
    elif sp == SINH:
        amp = 0.5 * L / math.sinh(0.5 * st)
        x = np.where(2 * np.arange(n + 1) <= n, amp * np.sinh(st * s), L - amp * np.sinh(st * (1.0 - s)))
    else:
        x = L * s
    x[0], x[-1] = 0.0, L
    return x


def _widths(n, L, sp, st):
    return np.diff(_faces(n, L, sp, st))


def _rb_params(n, H, Ra, sp):
    nu = 0.1 * H * math.sqrt(1.0 / Ra)
    tau = 3.0 * nu
    dt = 1.0 if sp == UNIFORM else 0.9 * min(1.0, _widths(n, H, sp, 2.0).min(), 8.0 * tau)
    return dict(tau=tau, tau_g=tau, dt=float(dt), beta=0.01 / H, grav=1.0, T0=1.0, T_bot=1.5, T_top=0.5)


def _rb3_params(case):
    nz, fv = case["nz"], case["scheme"] == "fv"
    tau = 0.5 if fv else 0.05
    return dict(tau=tau, tau_g=tau, dt=4.0 if fv else 1.0, beta=(1.325e-4 if fv else 1.325e-3) * 64.0 / nz, grav=1.0,
                T0=2.0, T_bot=3.0, T_top=1.0)


def _params(case):
    if case["kind"] == "rb":
        return _rb_params(case["ny"], float(case["ny"]), case["Ra"], case["sy"])
    if case["kind"] == "rb3":
        return _rb3_params(case)
    return dict(tau=case["tau"], dt=case["dt"], ax=case["ax"])


def _velocity(case, seed):
    """Three seeded vortex modes per axis (divergence-free, no slip on wall
    axes), of order case["u"]; plus the parabola on a channel."""
    rng = np.random.default_rng(seed)
    ax = []
    for n, sp, bc in ((case["nx"], case["sx"], case["bcx"]), (case["ny"], case["sy"], case["bcy"])):
        f = _faces(n, float(n), sp, case["stretch"])
        ax.append((0.5 * (f[1:] + f[:-1]) / n, bc))  # centres over the length

    def factor(x, m, bc, phase):  # a mode and its derivative over 2 pi m / L
        if bc == WALLS:
            return np.sin(math.pi * m * x) ** 2, 0.5 * np.sin(2.0 * math.pi * m * x)
        return np.sin(2.0 * math.pi * m * x + phase), np.cos(2.0 * math.pi * m * x + phase)

    u, v = np.zeros((case["ny"], case["nx"])), np.zeros((case["ny"], case["nx"]))
    ref = case["ny"] if case["nx"] < 8 else min(case["nx"], case["ny"])
    for m in (1, 2, 3):
        (xs, bx), (ys, by) = ax
        mx = 0 if case["nx"] < 8 else m
        sx, dx = factor(xs, mx, bx, rng.uniform(0, 2 * math.pi))
        sy, dy = factor(ys, m, by, rng.uniform(0, 2 * math.pi))
        amp = case["u"] * rng.uniform(0.5, 1.0) / m
        if case["kind"] == "channel":
            amp *= 0.1
        if mx == 0:
            sx, dx = np.ones_like(xs), np.zeros_like(xs)
        u += np.outer(dy, amp * ref / case["ny"] * sx)
        v -= np.outer(sy, amp * ref / case["nx"] * dx)
    if case["kind"] == "channel":
        y = ax[1][0]
        u += (4.0 * case["u"] * y * (1.0 - y))[:, None]
    return u, v


def _serve_requests(case, seed):
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["requests"]):
        # sizes over their whole range in every stream, in an order of its own
        t = (i + 0.5) / case["requests"]
        n = int(round(case["nmin"] * (case["nmax"] / case["nmin"]) ** t))
        steps = int(rng.integers(case["steps_lo"], case["steps_hi"] + 1))
        Ra = float(10 ** rng.uniform(4.0, 8.0))
        out.append(dict(n=n, steps=steps, seed=int(rng.integers(1, 2 ** 31)), p=_rb_params(n, float(n), Ra, TANH)))
    return [out[i] for i in rng.permutation(len(out))]


def _pinned(shape):
    return torch.empty(shape, dtype=torch.float64, pin_memory=torch.cuda.is_available())


def _ptr(t):
    return None if t is None else ctypes.cast(t.data_ptr(), ctypes.POINTER(ctypes.c_double))


def prepare(case, seed):
    if case["kind"] == "serve":
        return {"case": case, "requests": _serve_requests(case, seed)}
    thermal = case["kind"] in ("rb", "rb3")
    nx, ny = case["nx"], case["ny"]
    amp = 1e-3
    if case["kind"] == "rb3":
        nz, fv = case["nz"], case["scheme"] == "fv"
        k = 10.0 if fv else 1.0
        g = lb.Grid3(nx, ny, nz, lx=k * nx, ly=k * ny, lz=k * nz, sz=SINH if fv else UNIFORM,
                     stretch_z=4.0 if fv else 0.0, bcz=WALLS, thermal=True, store=case["store"])
        g.init(kind=lb.LB_INIT_RB, amp=amp, seed=seed, **_params(case))
        shape, q = (nz, ny, nx), 19
    else:
        g = lb.Grid(nx, ny, sx=case["sx"], sy=case["sy"], stretch_x=case["stretch"], stretch_y=case["stretch"],
                    bcx=case["bcx"], bcy=case["bcy"], thermal=thermal, store=case["store"])
        if thermal:
            g.init(kind=lb.LB_INIT_RB, amp=amp, seed=seed, **_params(case))
        else:
            u, v = _velocity(case, seed)
            g.init(kind=lb.LB_INIT_FIELDS, ux=u, uy=v, **_params(case))
        shape, q = (ny, nx), 9
    if case["out"] == "pops":
        out = {"f": _pinned((q,) + shape), "g": _pinned((q,) + shape) if thermal else None}
    else:
        names = ("rho", "ux", "uy") + (("uz",) if q == 19 else ()) + (("T",) if thermal else ())
        out = {k: _pinned(shape) for k in names}
    return {"case": case, "grid": g, "out": out}


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        return _run_serve(state)
    g, o = state["grid"], state["out"]
    (g.step_fv if case["scheme"] == "fv" else g.step_st)(case["steps"])
    api = lb.load()
    if case["kind"] == "rb3":
        st = (api.lb3_get_populations(g.handle, _ptr(o["f"]), _ptr(o["g"])) if case["out"] == "pops" else
              api.lb3_moments(g.handle, *(_ptr(o.get(k)) for k in ("rho", "ux", "uy", "uz", "T"))))
    else:
        st = (api.lb_get_populations(g.handle, _ptr(o["f"]), _ptr(o["g"])) if case["out"] == "pops" else
              api.lb_moments(g.handle, *(_ptr(o.get(k)) for k in ("rho", "ux", "uy", "T"))))
    if st != lb.LB_OK:
        raise lb.LBError(st, lb.lb_last_error())
    return {k: v for k, v in o.items() if v is not None}


def _run_serve(state):
    case = state["case"]
    s = lb.Server(store=case["store"], thermal=True)
    for i, r in enumerate(state["requests"]):
        s.submit(i, r["steps"], r["n"], r["n"], sy=TANH, stretch_y=2.0, bcy=WALLS, kind=lb.LB_INIT_RB, amp=1e-3,
                 seed=r["seed"], **r["p"])
    res = {}
    while len(res) < len(state["requests"]):
        s.pump()
        for r in s.results():
            res[r["id"]] = r
    s.close()
    order = range(len(state["requests"]))
    return {"status": np.array([res[i]["status"] for i in order]),
            "steps": np.array([res[i]["steps"] for i in order]),
            **{k: np.array([res[i][k] for i in order]) for k in ("nu_vol", "nu_bot", "nu_top", "mass")}}


# -------------------------------------------------------------------- work --

_BYTES = {"f64": 8, "f32": 4, "f16dev": 2, "bf16dev": 2}
# operations per cell update from the formulas of a step, shared terms once
# (an FMA counts two): D2Q9 as configs.flops_per_cell; D3Q19 by the same count
_FLOPS = {("fv", 9, False): 598, ("fv", 9, True): 926, ("st", 9, False): 173, ("st", 9, True): 220,
          ("fv", 19, True): 2200, ("st", 19, True): 480}


def work(case):
    """Each step reads and writes every population once; the results are
    written once more in FP64."""
    if case["kind"] == "serve":
        b = f = 0
        for r in _serve_requests(case, 0):
            c = r["n"] ** 2 * r["steps"]
            b += c * 36 * _BYTES[case["store"]]
            f += c * _FLOPS["fv", 9, True]
        return {"bytes": b, "flops": f}
    q = 19 if case["kind"] == "rb3" else 9
    th = case["kind"] in ("rb", "rb3")
    cells = case["nx"] * case["ny"] * case.get("nz", 1)
    pops = q * (2 if th else 1)
    outs = pops if case["out"] == "pops" else (4 if q == 19 else 3) + th
    return {"bytes": cells * (case["steps"] * 2 * pops * _BYTES[case["store"]] + 8 * outs),
            "flops": cells * case["steps"] * _FLOPS[case["scheme"], q, th]}


# ------------------------------------------------------------------- exact --

_C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_W2 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
_C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
       (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
       (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_W3 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _splitmix(seed, n):
    """U in [0, 1) of counters 0..n-1 (SplitMix64 from state seed ^ counter)."""
    with np.errstate(over="ignore"):
        z = (np.uint64(seed) ^ np.arange(n, dtype=np.uint64)) + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z ^= z >> np.uint64(31)
    return (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


class _Exact:
    """The FV (semi-implicit, Heun, QUICK) and ST steps in FP64.  Fields are
    [..., y, x]; axis k is tensor dimension -1 - k; the last axis has gravity
    and, on a thermal layer, the plates."""

    def __init__(self, n, L, sp, st, bc, thermal, tau, dt, tau_g=None, ax=0.0, beta=0.0, grav=0.0, T0=1.0, T_bot=1.0,
                 T_top=1.0):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.D = len(n)
        self.c, self.w = (_C2, _W2) if self.D == 2 else (_C3, _W3)
        self.Q = len(self.w)
        self.inv = [self.c.index(tuple(-x for x in v)) for v in self.c]
        self.n, self.L, self.bc, self.th = n, L, bc, thermal
        self.tau, self.dt, self.taug = tau, dt, tau if tau_g is None else tau_g
        self.a0 = [ax] + [0.0] * (self.D - 1)
        self.bg, self.T0, self.Tb, self.Tt = beta * grav, T0, T_bot, T_top
        self.cen, self.wid, self.wp, self.wm = [], [], [], []
        for k in range(self.D):
            x = _faces(n[k], L[k], sp[k], st[k])
            c = 0.5 * (x[1:] + x[:-1])
            if bc[k] == PERIODIC:
                i = np.arange(-2, n[k] + 2)
                p = c[i % n[k]] + (i // n[k]) * L[k]
            else:
                p = np.concatenate([[-c[1], -c[0]], c, [2 * L[k] - c[-1], 2 * L[k] - c[-2]]])
            self.cen.append(c)
            self.wid.append(self._vec(np.diff(x), k))
            # Lagrange weights at every face for the nodes from k - 2 and from k - 1
            for lst, o in ((self.wp, 0), (self.wm, 1)):
                a, b, d = p[o:o + n[k] + 1], p[o + 1:o + n[k] + 2], p[o + 2:o + n[k] + 3]
                lst.append([self._vec(v, k) for v in ((x - b) * (x - d) / ((a - b) * (a - d)),
                                                      (x - a) * (x - d) / ((b - a) * (b - d)),
                                                      (x - a) * (x - b) / ((d - a) * (d - b)))])

    def _vec(self, v, k):
        return torch.as_tensor(v, dtype=torch.float64, device=self.dev).reshape((-1,) + (1,) * k)

    def _macro(self, f, g, hf):
        rho = f.sum(0)
        T = g.sum(0) if self.th else None
        a = list(self.a0)
        if self.th:
            a[-1] = self.a0[-1] + self.bg * (T - self.T0)
        u = []
        for k in range(self.D):
            j = None
            for q in range(self.Q):
                if self.c[q][k]:
                    t = f[q] if self.c[q][k] > 0 else -f[q]
                    j = t.clone() if j is None else j.add_(t)
            u.append(j.div_(rho).add_(hf * a[k]))
        return rho, u, T, a

    def _terms(self, m):
        """Per population: f_eq, F and f_eq / rho; nothing is kept over populations."""
        rho, u, T, a = m
        uu = sum(x * x for x in u).mul_(1.5)
        force = self.th or any(self.a0)
        ua = sum(x * y for x, y in zip(u, a)) if force else None
        for q in range(self.Q):
            c, w = self.c[q], self.w[q]
            cu = sum((x if s > 0 else -x) for x, s in zip(u, c) if s) if any(c) else None
            e = -uu if cu is None else cu * (3.0 + 4.5 * cu) - uu
            e = e.add_(1.0).mul_(w)
            F = None
            if force:
                F = -3.0 * ua
                if cu is not None:
                    ca = sum(s * x for s, x in zip(c, a))
                    F = F + 3.0 * ca + 9.0 * cu * ca
                F = F.mul_(rho).mul_(w)
            yield q, e * rho, F, e

    def start(self, rho, u, T):
        dt = self.dt
        a = list(self.a0)
        if self.th:
            a[-1] = self.a0[-1] + self.bg * (T - self.T0)
        shape = tuple(reversed(self.n))
        f = torch.empty((self.Q,) + shape, dtype=torch.float64, device=self.dev)
        g = torch.empty_like(f) if self.th else None
        for q, feq, F, e in self._terms((rho, u, T, a)):
            f[q] = feq if F is None else feq - 0.5 * dt * F
            if self.th:
                g[q] = e * T
        return f, g

    def start_rb(self, seed, amp):
        n, H = self.n, self.L[-1]
        y, wid = self.cen[-1], self.wid[-1].cpu().numpy().ravel()
        dT = self.Tb - self.Tt
        b = np.exp(3.0 * self.bg * dT * (0.5 * y - 0.5 * y * y / H))
        rho = self._vec(b * H / (wid * b).sum(), self.D - 1).expand(tuple(reversed(n))).contiguous()
        U = torch.as_tensor(_splitmix(seed, int(np.prod(n))), device=self.dev).reshape(tuple(reversed(n)))
        T = self._vec(self.T0 + dT * (0.5 - y / H), self.D - 1) + amp * dT * (2.0 * U - 1.0)
        return self.start(rho, [torch.zeros_like(rho) for _ in range(self.D)], T)

    def _ghosts(self, h, q, k, plates):
        """Population q of h with two ghost layers on axis k."""
        d = h.dim() - 2 - k  # dimension of h[q]
        n = self.n[k]

        def take(b, i):
            return h[b].select(d, i).unsqueeze(d)
        if self.bc[k] == PERIODIC:
            idx = [take(q, -2 % n), take(q, -1 % n)], [take(q, 0), take(q, 1 % n)]
        else:
            b, w = self.inv[q], 2.0 * self.w[q]
            lo, hi = [take(b, 1), take(b, 0)], [take(b, n - 1), take(b, n - 2)]
            if plates:
                lo, hi = [w * self.Tb - v for v in lo], [w * self.Tt - v for v in hi]
            idx = lo, hi
        return torch.cat(idx[0] + [h[q]] + idx[1], d), d

    def _advect(self, h, q, plates):
        out = None
        for k in range(self.D):
            c = self.c[q][k]
            if not c:
                continue
            p, d = self._ghosts(h, q, k, plates)
            n, (w, o) = self.n[k], (self.wp[k], 0) if c > 0 else (self.wm[k], 1)
            phi = w[0] * p.narrow(d, o, n + 1)
            phi.addcmul_(w[1].expand_as(phi), p.narrow(d, o + 1, n + 1))
            phi.addcmul_(w[2].expand_as(phi), p.narrow(d, o + 2, n + 1))
            t = (phi.narrow(d, 1, n) - phi.narrow(d, 0, n)).div_(self.wid[k])
            if c < 0:
                t.neg_()
            out = t if out is None else out.add_(t)
        return out

    def _fields(self, f, g):
        """The advected fields h, hg of Eq. (semi)."""
        dt = self.dt
        o, og = dt / (2.0 * self.tau + dt), dt / (2.0 * self.taug + dt)
        hF = 0.5 * dt * (1.0 - o)
        m = self._macro(f, g, 0.5 * dt)
        h = torch.empty_like(f)
        hg = torch.empty_like(g) if self.th else None
        for q, feq, F, e in self._terms(m):
            torch.lerp(f[q], feq, o, out=h[q])
            if F is not None:
                h[q].add_(F, alpha=hF)
            if self.th:
                torch.lerp(g[q], e * m[2], og, out=hg[q])
        return h, hg

    def fv(self, f, g):
        dt = self.dt
        h, hg = self._fields(f, g)
        base, star = [], []
        for p, hh in ((f, h), (g, hg)):
            if p is None:
                base.append(None)
                star.append(None)
                continue
            b = 2.0 * hh - p  # f~ + Coll
            s = b.clone()
            for q in range(self.Q):
                adv = self._advect(hh, q, p is g)
                if adv is not None:
                    b[q].add_(adv, alpha=-0.5 * dt)
                    s[q].add_(adv, alpha=-dt)
            base.append(b)
            star.append(s)
        del h, hg
        hs, hgs = self._fields(*star)
        for b, hh in ((base[0], hs), (base[1], hgs)):
            if b is None:
                continue
            for q in range(self.Q):
                adv = self._advect(hh, q, b is base[1])
                if adv is not None:
                    b[q].add_(adv, alpha=-0.5 * dt)
        return base[0], base[1]

    def st(self, f, g):
        o, og = 1.0 / (self.tau + 0.5), 1.0 / (self.taug + 0.5)
        m = self._macro(f, g, 0.5)
        nf = torch.empty_like(f)
        ng = torch.empty_like(g) if self.th else None
        bounce = []
        for q, feq, F, e in self._terms(m):
            post = torch.lerp(f[q], feq, o)
            if F is not None:
                post.add_(F, alpha=1.0 - 0.5 * o)
            sets = [(nf, post, False)]
            if self.th:
                sets.append((ng, torch.lerp(g[q], e * m[2], og), True))
            c = self.c[q]
            dims = [post.dim() - 1 - k for k in range(self.D) if c[k]]
            move = [c[k] for k in range(self.D) if c[k]]
            for dst, v, plates in sets:
                r = torch.roll(v, move, dims) if dims else v
                dst[q] = r
            # half-way bounce-back on wall axes (the plates: anti-bounce-back of g)
            for k in range(self.D):
                if not c[k] or self.bc[k] == PERIODIC:
                    continue
                i = self.n[k] - 1 if c[k] > 0 else 0
                d = post.dim() - 1 - k
                bounce.append((q, d, i, [(dst, v.select(d, i).clone(), plates) for dst, v, plates in sets]))
        for q, d, i, sets in bounce:
            b = self.inv[q]
            for dst, v, plates in sets:
                tw = self.Tb if i == 0 else self.Tt
                dst[b].select(d, i).copy_(2.0 * self.w[q] * tw - v if plates else v)
        return nf, ng

    def observe(self, f, g):
        rho, u, T, _ = self._macro(f, g, 0.5 * self.dt)
        return rho, u, T

    def nusselt(self, f, g):
        """Volume and plate Nusselt numbers, and the mass (2-D layer)."""
        rho, u, T = self.observe(f, g)
        H, dT, V = self.L[-1], self.Tb - self.Tt, self.wid[0] * self.wid[1]
        vol = 1.0 + H * float((V * u[-1] * (T - self.T0)).sum() / V.sum()) / (self.taug / 3.0 * dT)
        Tm = ((T * self.wid[0]).sum(-1) / self.L[0]).tolist()
        y = self.cen[-1]

        def grad(z0, z1, Tw, t0, t1):  # parabola through the wall and two nodes
            return -(z0 + z1) / (z0 * z1) * Tw + z1 / (z0 * (z1 - z0)) * t0 - z0 / (z1 * (z1 - z0)) * t1
        bot = -H * grad(y[0], y[1], self.Tb, Tm[0], Tm[1]) / dT
        top = H * grad(H - y[-1], H - y[-2], self.Tt, Tm[-1], Tm[-2]) / dT
        return vol, bot, top, float((V * rho).sum())


def exact(case, seed):
    if case["kind"] == "serve":
        reqs = _serve_requests(case, seed)
        if sum(r["steps"] for r in reqs) > 2000:
            return None
        vals = []
        for r in reqs:
            n = r["n"]
            X = _Exact((n, n), (float(n), float(n)), (UNIFORM, TANH), (0.0, 2.0), (PERIODIC, WALLS), True, **r["p"])
            f, g = X.start_rb(r["seed"], 1e-3)
            for _ in range(r["steps"]):
                f, g = X.fv(f, g)
            vals.append(X.nusselt(f, g))
        cols = np.array(vals).T
        return {"status": None, "steps": None, "nu_vol": cols[0], "nu_bot": cols[1], "nu_top": cols[2],
                "mass": cols[3]}
    nx, ny = case["nx"], case["ny"]
    if nx * ny * case.get("nz", 1) * case["steps"] > 1.4e10:
        return None
    if case["kind"] == "rb3":
        fv, nz = case["scheme"] == "fv", case["nz"]
        k = 10.0 if fv else 1.0
        X = _Exact((nx, ny, nz), (k * nx, k * ny, k * nz), (UNIFORM, UNIFORM, SINH if fv else UNIFORM),
                   (0.0, 0.0, 4.0), (PERIODIC, PERIODIC, WALLS), True, **_params(case))
        f, g = X.start_rb(seed, 1e-3)
    else:
        th = case["kind"] == "rb"
        X = _Exact((nx, ny), (float(nx), float(ny)), (case["sx"], case["sy"]), (case["stretch"],) * 2,
                   (case["bcx"], case["bcy"]), th, **_params(case))
        if th:
            f, g = X.start_rb(seed, 1e-3)
        else:
            u, v = (torch.as_tensor(x, device=X.dev) for x in _velocity(case, seed))
            f, g = X.start(torch.ones_like(u), [u, v], None)
    step = X.fv if case["scheme"] == "fv" else X.st
    for _ in range(case["steps"]):
        f, g = step(f, g)
    if case["out"] == "pops":
        return {"f": f.cpu(), **({"g": g.cpu()} if g is not None else {})}
    rho, u, T = X.observe(f, g)
    out = {"rho": rho, "ux": u[0], "uy": u[1]}
    if X.D == 3:
        out["uz"] = u[2]
    if T is not None:
        out["T"] = T
    return {k: v.cpu() for k, v in out.items()}
