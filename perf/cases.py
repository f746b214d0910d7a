"""Workloads of the solver that its speed is measured on.

Every case is a piece of work that a program using the package does through its public entry points: runs of some
steps on 2D and 3D boxes in both precisions, with the state on the device or in host memory, the job of a batched
ensemble, a gradient by the adjoint, and an analysis of a state.  Inputs are fields of developed convection made from
the seed alone (the hydrostatic profile under rolls of random phase plus grid-scale noise); `exact` steps them in
float64 with plain torch operations, written from the equations and the scheme and not from the package.

The library keeps one solver context per process, so the states of one case share a context: each holds an initial
condition, and a pass starts from it.
"""
import math

import numpy as np
import torch

import paper_2411_10372_gb300 as cm

EPS = 0.1


# ---- the cases --------------------------------------------------------------------------------------------------------

def _run(name, nx, nz, *, ny=1, prec="fp32", via="device", steps, Ra, Pr=1.0, gamma=5.0 / 3.0, D=0.5, aspect=4.0,
         zstretch=0.0, diag_every=0):
    return {"name": name, "kind": "run", "prec": prec, "via": via, "ndim": 3 if ny > 1 else 2, "nx": nx, "ny": ny,
            "nz": nz, "steps": steps, "Ra": Ra, "Pr": Pr, "gamma": gamma, "D": D, "aspect": aspect,
            "zstretch": zstretch, "diag_every": diag_every}


def listed():
    return [
        # the smallest box that is run in earnest: launches and latency.  Short, like every float32 run here: a smooth
        # developed flow multiplies a rounding error by a thousand within a hundred steps
        _run("box_128x64_fp32", 128, 64, via="host", steps=10, Ra=1e6, Pr=0.7, D=0.49, aspect=2.0),
        # the parity workload in float64, a small box as well
        _run("box_256x64_fp64", 256, 64, prec="fp64", via="host", steps=100, Ra=1e6),
        # an odd number of columns and an odd number of planes
        _run("odd_1001x301_fp32", 1001, 301, steps=20, Ra=1e8),
        # the tanh grid of the 2D production run at Ra = 1e9
        _run("tanh_3000x1501_fp32", 3000, 1501, steps=20, Ra=1e9, Pr=0.7, gamma=1.3, zstretch=1.0),
        # the headline box
        _run("box_4096x1024_fp32", 4096, 1024, steps=25, Ra=1e10),
        # the same box in float64
        _run("box_4096x1024_fp64", 4096, 1024, prec="fp64", steps=2, Ra=1e10),
        # the 3D box
        _run("box_512x512x128_fp32", 512, 128, ny=512, steps=5, Ra=1e9),
        # the 3D production run at Ra = 1e8 on its tanh grid, at half resolution
        _run("tanh_256x256x128_fp32", 256, 128, ny=256, steps=10, Ra=1e8, Pr=0.7, gamma=1.3, zstretch=1.2),
        # a small 3D box in float64, odd in every direction
        _run("box_97x81x49_fp64", 97, 49, ny=81, prec="fp64", steps=5, Ra=1e6),
        # the job of a batched ensemble: 64 uneven boxes set up, stepped, sampled and read back
        {"name": "batch_64", "kind": "batch", "nbox": 64, "nz_min": 32, "nz_max": 256, "sizes": 2024, "steps": 600,
         "zstretch": 0.0},
        # gradient of a window mean of the plate Nusselt number: forward and backward
        {"name": "adjoint_1024x256", "kind": "adjoint", "nx": 1024, "nz": 256, "Ra": 1e8, "steps": 40, "K": 10,
         "win": 31, "zstretch": 0.0},
        # the analyses of a float32 state
        {"name": "analysis_4096x1024", "kind": "analysis", "ndim": 2, "prec": "fp32", "nx": 4096, "ny": 1, "nz": 1024,
         "Ra": 1e10, "bins": 96, "zstretch": 0.0},
    ]


def _spread(rng, lo, hi):
    """An integer between lo and hi, uniform in its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _stable_Ra(rng, nz, zstretch):
    """A Rayleigh number that the explicit scheme resolves on nz planes, to two decades above the least."""
    return 1e6 * (nz / 64.0) ** 2 * (8.0 if zstretch > 1.2 else 3.0) * 10.0 ** rng.uniform(0.0, 2.0)


def draw(rng):
    kind = rng.choices(["2d32", "2d64", "3d32", "3d64", "batch", "adjoint", "analysis"], [10, 4, 4, 2, 2, 2, 2])[0]
    zs = rng.choice([0.0, 0.0, rng.uniform(0.5, 2.0)])
    if kind == "batch":
        nz_min = _spread(rng, 16, 64)
        return {"kind": "batch", "nbox": rng.randint(4, 64), "nz_min": nz_min, "nz_max": nz_min * rng.randint(1, 4),
                "sizes": rng.randrange(1 << 20), "steps": rng.randint(100, 300), "zstretch": min(zs, 1.0)}
    if kind == "adjoint":
        nz = _spread(rng, 24, 256)
        nx, steps = _spread(rng, nz, 4 * nz), rng.randint(8, 40)
        return {"kind": "adjoint", "nx": nx, "nz": nz, "Ra": _stable_Ra(rng, nz, zs), "steps": steps,
                "K": rng.choice([0, rng.randint(1, steps)]), "win": rng.randint(1, steps), "zstretch": zs}
    if kind == "analysis":
        nz = _spread(rng, 33, 1024)
        return {"kind": "analysis", "ndim": 2, "prec": rng.choice(["fp32", "fp64"]), "nx": _spread(rng, nz, 4 * nz),
                "ny": 1, "nz": nz, "Ra": _stable_Ra(rng, nz, zs), "bins": rng.randint(8, 200), "zstretch": zs}
    if kind in ("3d32", "3d64"):
        nz = _spread(rng, 17, 128 if kind == "3d32" else 64)
        nx, ny = _spread(rng, nz, 4 * nz), _spread(rng, nz, 4 * nz)
        most = 1e8 if kind == "3d32" else 4e6
    else:
        nz = _spread(rng, 33, 1500 if kind == "2d32" else 600)
        nx, ny = _spread(rng, nz, 4 * nz), 1
        most = 2e8 if kind == "2d32" else 1e7
    steps = max(2, min(rng.randint(5, 25) if kind.endswith("32") else rng.randint(20, 100), int(most / (nx * ny * nz))))
    if rng.random() < 0.5:  # half the sizes even, half as they come
        nx += nx & 1
    return {k: v for k, v in _run("", nx, nz, ny=ny, prec="fp64" if kind.endswith("64") else "fp32",
                                  via=rng.choice(["device", "device", "host"]) if ny == 1 else "device", steps=steps,
                                  diag_every=rng.choice([0, 10]), Ra=_stable_Ra(rng, nz, zs), Pr=rng.choice([0.7, 1.0]),
                                  gamma=rng.choice([1.3, 1.4, 5.0 / 3.0]), zstretch=zs).items() if k != "name"}


# ---- equations: closures, planes, initial conditions ------------------------------------------------------------------

class _Model:
    """Coefficients and planes of a case (nondimensional equations; FP64)."""

    def __init__(self, case, device):
        get = case.get
        self.Ra, self.Pr = case["Ra"], get("Pr", 1.0)
        self.gamma, self.D, self.aspect = get("gamma", 5.0 / 3.0), get("D", 0.5), get("aspect", 4.0)
        self.nx, self.ny, self.nz, self.ndim = case["nx"], get("ny", 1), case["nz"], get("ndim", 2)
        self.a = (self.gamma - 1.0) / (self.gamma * EPS * self.D)
        self.b = self.gamma * EPS * self.D
        self.g = 1.0 / EPS
        self.cs2 = self.gamma * self.a
        self.t_top = 1.0 - EPS - self.D
        K = self.nz - 1
        z = np.arange(self.nz) / K
        beta = get("zstretch", 0.0)
        if beta > 0:
            z = 0.5 * (1.0 + np.tanh(beta * (2.0 * np.arange(self.nz) / K - 1.0)) / np.tanh(beta))
            z[0], z[K] = 0.0, 1.0
        self.planes = z
        self.hmin = min(self.aspect / self.nx, float(np.min(np.diff(z))))
        if self.ndim == 3:
            self.hmin = min(self.hmin, self.aspect / self.ny)
        col = lambda v: torch.tensor(v, dtype=torch.float64, device=device)[:, None, None]  # noqa: E731
        self.z, hp = col(z), np.diff(z)
        w = np.concatenate([hp[:1] / 2, (hp[:-1] + hp[1:]) / 2, hp[-1:] / 2])
        self.hp, self.w, self.span = col(hp), col(w), col(hp[:-1] + hp[1:])
        near = np.concatenate([hp[:1], np.minimum(hp[:-1], hp[1:]), hp[-1:]])
        self.h_cfl = col(near)
        self.h = {"x": self.aspect / self.nx, "y": self.aspect / self.ny}
        self.axes = ["x", "y", "z"] if self.ndim == 3 else ["x", "z"]
        self.mu, self.kth = math.sqrt(self.Pr / self.Ra), 1.0 / (EPS * self.D * math.sqrt(self.Ra * self.Pr))
        self.device = device

    def profile(self):
        """Temperature and pressure of the conduction state on the planes."""
        T = 1.0 - (1.0 - self.t_top) * self.z
        return T, self.a * T ** (self.g / (self.a * (1.0 - self.t_top)))

    def fixed_dt(self):
        """A time step below the CFL limit of every state that `_field` makes."""
        return 0.45 * self.hmin / (math.sqrt(self.cs2 * 1.06) + 0.8)


def _field(model, seed, dtype):
    """Developed convection: rolls of a few random modes in velocity and temperature, grid-scale noise of amplitude
    1e-3 in temperature, on the hydrostatic profile; plates at rest and at their temperatures.  (nf, nz, ny, nx)."""
    m, dev = model, model.device
    g = torch.Generator(device="cpu").manual_seed(int(seed) & 0x7FFFFFFF)
    x = torch.arange(m.nx, device=dev, dtype=torch.float64)[None, None, :] * (2 * math.pi / m.nx)
    y = torch.arange(m.ny, device=dev, dtype=torch.float64)[None, :, None] * (2 * math.pi / m.ny)

    def rolls(amplitude):
        f = torch.zeros((m.nz, m.ny, m.nx), dtype=torch.float64, device=dev)
        for r in torch.rand((5, 5), generator=g, dtype=torch.float64).tolist():
            kx, ky, kz = 1 + int(6 * r[0]), int(6 * r[1]) if m.ndim == 3 else 0, 1 + int(3 * r[2])
            f += torch.sin(math.pi * kz * m.z) * torch.cos(kx * x + ky * y + 2 * math.pi * r[3]) * (0.5 + r[4])
        return f * (amplitude / 5)

    T, p = m.profile()
    noise = torch.rand((m.nz, m.ny, m.nx), generator=torch.Generator(device=dev).manual_seed(int(seed) & 0x7FFFFFFF),
                       dtype=torch.float32, device=dev).double()
    T = T + rolls(0.05) + (2e-3 * noise - 1e-3)
    T[0], T[-1] = 1.0, m.t_top
    rho = p / (m.a * T)
    u = [rolls(0.3) for _ in m.axes]
    for v in u:
        v[0], v[-1] = 0.0, 0.0
    E = rho * (0.5 * sum(v * v for v in u) + T / m.b + m.g * m.z)
    return torch.stack([rho, *(rho * v for v in u), E]).to(dtype)


# ---- the library's side -----------------------------------------------------------------------------------------------

_now = {"key": None, "solver": None, "buf": None}  # the process's one context, and the case that it was made for


def _context(case, **params):
    """The solver context of a case; made when the last one was another case's."""
    key = repr(sorted((k, v) for k, v in case.items() if k not in ("name", "steps")))
    if _now["key"] != key:
        if _now["solver"] is not None:
            _now["solver"].close()
        _now.update(key=None, solver=None, buf=None)
        grid = cm.cm_grid(case["ndim"], case["nx"], case["ny"], case["nz"], case.get("aspect", 4.0),
                          case["zstretch"], None)
        prec = cm.CM_FP64 if case["prec"] == "fp64" else cm.CM_FP32
        buf = torch.zeros(cm.cm_state_bytes(grid, prec), dtype=torch.uint8, device="cuda")
        solver = cm.Solver(case["nx"], case["nz"], case["Ra"], case.get("Pr", 1.0), case.get("gamma", 5.0 / 3.0),
                           ny=case["ny"], ndim=case["ndim"], aspect=case.get("aspect", 4.0), precision=case["prec"],
                           zstretch=case["zstretch"], D=case.get("D", 0.5), state_buf=buf.data_ptr(), **params)
        _now.update(key=key, solver=solver, buf=buf)
    return _now["solver"]


def _state_view(case):
    """The context's current state as a torch tensor (nf, nz, ny, nx) on the caller's own state buffer."""
    pitch, nf, elem = cm.cm_state_layout()
    at = (cm.cm_state_ptr(0) - _now["buf"].data_ptr()) // elem
    flat = _now["buf"].view(torch.float64 if elem == 8 else torch.float32)
    rows = case["nz"] * case["ny"]
    return flat[at: at + nf * rows * pitch].view(nf, case["nz"], case["ny"], pitch)[..., :case["nx"]]


def _boxes(case):
    """Grids and Rayleigh numbers of an ensemble: planes spread over their logarithm, four times as many columns."""
    r = np.random.default_rng(case["sizes"])
    nz = np.round(case["nz_min"] * (case["nz_max"] / case["nz_min"]) ** r.random(case["nbox"])).astype(int)
    Ra = 10.0 ** (5.0 + 4.0 * r.random(case["nbox"]))
    Ra = np.maximum(Ra, 40.0 * nz.astype(float) ** 2 * (1.0 if case["zstretch"] == 0 else 4.0))  # resolved explicitly
    return [(4 * int(n), int(n)) for n in nz], [float(v) for v in Ra]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        sizes, Ra = _boxes(case)
        params = cm.cm_default_params()
        params.precision, params.seed = cm.CM_FP32, int(seed)
        grids = [cm.cm_grid(2, nx, 1, nz, 4.0, case["zstretch"], None) for nx, nz in sizes]
        return {"case": case, "grids": grids, "Ra": Ra, "params": params, "sizes": sizes}
    model = _Model(case, "cuda")
    if kind == "adjoint":
        X = _field(model, seed, torch.float64)[:, :, 0].contiguous()
        grid = {"nx": case["nx"], "nz": case["nz"], "zstretch": case["zstretch"],
                "adj_limiter": cm.CM_ADJ_PHI_FROZEN}
        return {"case": case, "X": X, "Ra": torch.tensor(case["Ra"], dtype=torch.float64), "grid": grid}
    dtype = torch.float64 if case["prec"] == "fp64" else torch.float32
    X = _field(model, seed, dtype)
    if kind == "run" and case["via"] == "host":
        _context(case, diag_every=case["diag_every"])
        shape = X.shape if case["ndim"] == 3 else X[:, :, 0].shape
        host = torch.empty(shape, dtype=dtype, pin_memory=True)
        host.copy_(X.view(shape))
        return {"case": case, "in": host.numpy(), "out": torch.empty(shape, dtype=dtype, pin_memory=True).numpy()}
    _context(case, dt_fixed=model.fixed_dt() if kind == "run" else 0.0, diag_every=case.get("diag_every", 0))
    return {"case": case, "X": X}


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        cm.cm_batch_init(state["grids"], state["Ra"], 1.0, 5.0 / 3.0, state["params"])
        cm.cm_batch_step(case["steps"])
        records = cm.cm_batch_diagnostics()
        X = [cm.cm_batch_get_state(b, np.empty((4, nz, nx))).astype(np.float32).ravel()
             for b, (nx, nz) in enumerate(state["sizes"])]
        cm.cm_batch_finalize()
        return {"X": np.concatenate(X), "energy": np.float32([r["energy"] for r in records]),
                "t": np.float32([r["t"] for r in records])}
    if case["kind"] == "adjoint":
        from paper_2411_10372_gb300.adjoint import NuObjective
        _now.update(key=None, solver=None, buf=None)  # the objective makes a context of its own
        X, Ra = state["X"].clone().requires_grad_(), state["Ra"].clone().requires_grad_()
        J = NuObjective.apply(X, Ra, state["grid"], case["steps"], case["K"], case["win"])
        J.backward()
        return {"J": J, "dX": X.grad, "dRa": Ra.grad}
    if case["kind"] == "analysis":
        _state_view(case).copy_(state["X"])
        profiles = cm.cm_ext_profiles(case["nz"])
        ext, hist = cm.cm_extended(case["bins"], -10.0, 0.0)
        return {"profiles": profiles, "hist": hist, "C": ext["C"], "r_max": ext["r_max"]}
    if case["via"] == "host":
        if case["prec"] == "fp64":
            record = cm.cm_run_host(state["in"], case["steps"], state["out"])
        else:
            record = cm.cm_run_host_f32(state["in"], case["steps"], state["out"])
        seen = cm.cm_diagnostics(1024) if case["diag_every"] else []
        return {"X": state["out"], "energy": [r["energy"] for r in seen + [record]],
                "KE": [r["KE"] for r in seen + [record]]}
    _state_view(case).copy_(state["X"])
    cm.cm_step(case["steps"])
    seen = cm.cm_diagnostics(1024) if case["diag_every"] else []
    return {"X": _state_view(case), "energy": [r["energy"] for r in seen], "KE": [r["KE"] for r in seen]}


# ---- the least work ---------------------------------------------------------------------------------------------------

# floating-point operations of the scheme per node and sweep (an add, a multiply, a divide, a square root count one)
_FLOPS = {2: 174, 3: 240}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        nodes = sum(nx * nz for nx, nz in _boxes(case)[0])
        return {"bytes": case["steps"] * nodes * 32.0, "flops": case["steps"] * nodes * 4.0 * _FLOPS[2]}
    nodes = case["nx"] * case.get("ny", 1) * case["nz"]
    if kind == "adjoint":  # the forward steps and, at three times their operations, the reverse ones
        return {"bytes": case["steps"] * nodes * 5 * 32.0, "flops": case["steps"] * nodes * 16.0 * _FLOPS[2]}
    elem = 8 if case["prec"] == "fp64" else 4
    if kind == "analysis":  # two calls
        return {"bytes": 2.0 * nodes * 4 * elem, "flops": 2.0 * nodes * 90}
    nf = 2 + case["ndim"]
    return {"bytes": case["steps"] * nodes * 2.0 * nf * elem,
            "flops": case["steps"] * nodes * 2.0 * case["ndim"] * _FLOPS[case["ndim"]]}


# ---- the same in float64 with plain torch operations ------------------------------------------------------------------

_DIM = {"x": 2, "y": 1, "z": 0}


def _primitives(m, X):
    u = {a: X[1 + i] / X[0] for i, a in enumerate(m.axes)}
    T = m.b * (X[-1] / X[0] - 0.5 * sum(v * v for v in u.values()) - m.g * m.z)
    return u, T, m.a * X[0] * T


def _one_sided(m, f, axis, forward):
    """Difference quotient to the next (forward) or from the last node; along z zero where there is none."""
    if axis != "z":
        return ((torch.roll(f, -1, _DIM[axis]) - f) if forward else (f - torch.roll(f, 1, _DIM[axis]))) / m.h[axis]
    d, pad = (f[1:] - f[:-1]) / m.hp, torch.zeros_like(f[:1])
    return torch.cat([d, pad] if forward else [pad, d])


def _central(m, f, axis):
    if axis != "z":
        return (torch.roll(f, -1, _DIM[axis]) - torch.roll(f, 1, _DIM[axis])) / (2.0 * m.h[axis])
    pad = torch.zeros_like(f[:1])
    return torch.cat([pad, (f[2:] - f[:-2]) / m.span, pad])


def _flux(m, X, along, forward, mu, kth):
    """F_along: [m_a; m_i u_a - tau_ia + p delta_ia; u_a (E + p) - K d_a T - u_i tau_ia]."""
    u, T, p = _primitives(m, X)
    d = lambda f, axis: _one_sided(m, f, axis, forward) if axis == along else _central(m, f, axis)  # noqa: E731
    div = sum(d(u[a], a) for a in m.axes)
    F, heat = [], -kth * d(T, along)
    for i, a in enumerate(m.axes):
        tau = mu * (2.0 * d(u[a], a) - 2.0 / 3.0 * div) if a == along else mu * (d(u[a], along) + d(u[along], a))
        F.append(X[1 + i] * u[along] - tau + (p if a == along else 0.0))
        heat = heat - u[a] * tau
    return torch.stack([X[1 + m.axes.index(along)], *F, u[along] * (X[-1] + p) + heat])


def _sweep(m, X, along, delta, mu, kth, frozen):
    """L_along(delta): predictor, corrector, their mean and the TVD term; conservative on uneven planes."""
    dim, periodic = 1 + _DIM[along], along != "z"
    up = lambda f: torch.roll(f, -1, dim)  # noqa: E731
    down = lambda f: torch.roll(f, 1, dim)  # noqa: E731
    at = 1 + m.axes.index("z")

    def plates(rho):
        """A state's two plates with densities rho: at rest, at their temperatures."""
        zero = torch.zeros_like(rho)
        T = torch.tensor([1.0, m.t_top], dtype=torch.float64, device=rho.device)[:, None, None]
        z = torch.tensor([0.0, 1.0], dtype=torch.float64, device=rho.device)[:, None, None]
        return torch.stack([rho, *[zero] * m.ndim, rho * (T / m.b + m.g * z)])

    F = _flux(m, X, along, True, mu, kth)
    if periodic:
        lam = delta / m.h[along]
        P = X - lam * (F - down(F))
        P = torch.cat([X[:, :1], P[:, 1:-1], X[:, -1:]], 1)
        FP = _flux(m, P, along, False, mu, kth)
        mean = 0.5 * (P + X - lam * (up(FP) - FP))
    else:
        lam = delta / m.w
        source = torch.zeros_like(X)
        source[at] = -m.g * X[0]
        P = X[:, 1:-1] - lam[1:-1] * (F[:, 1:-1] - F[:, :-2]) + delta * source[:, 1:-1]
        ends = plates(torch.stack([X[0, 0] - lam[0] * F[0, 0], X[0, -1] + lam[-1] * F[0, -2]]))
        P = torch.cat([ends[:, :1], P, ends[:, 1:]], 1)
        FP = _flux(m, P, along, False, mu, kth)
        source = torch.zeros_like(X)
        source[at] = -m.g * P[0]
        C = X[:, 1:-1] - lam[1:-1] * (FP[:, 2:] - FP[:, 1:-1]) + delta * source[:, 1:-1]
        rho = torch.stack([P[0, 0] + X[0, 0] - lam[0] * FP[0, 1], P[0, -1] + X[0, -1]])
        ends = plates(0.5 * rho)
        mean = torch.cat([ends[:, :1], 0.5 * (P[:, 1:-1] + C), ends[:, 1:]], 1)
    # TVD flux through the interface above each node
    u, T, _ = _primitives(m, X)
    speed = u[along].abs() + torch.sqrt(m.cs2 * T)
    if periodic:
        d0 = up(X) - X
        dm, dp, A0, A1, h = down(d0), up(d0), speed, torch.roll(speed, -1, _DIM[along]), m.h[along]
    else:  # interfaces of interior nodes alone
        d = X[:, 1:] - X[:, :-1]
        dm, d0, dp, A0, A1, h = d[:, :-2], d[:, 1:-1], d[:, 2:], speed[1:-2], speed[2:-1], m.hp[1:-1]
    dot = lambda p, q: sum(p[c] * q[c] for c in range(len(p)))  # noqa: E731
    sp, sm, dd = dot(dm, d0), dot(d0, dp), dot(d0, d0)
    if frozen:
        sp, sm, dd = sp.detach(), sm.detach(), dd.detach()
    flat = dd == 0
    safe = torch.where(flat, torch.ones_like(dd), dd)
    phi = lambda r: torch.clamp(2.0 * r, 0.0, 1.0)  # noqa: E731
    Co = delta * torch.where(A0 >= A1, A0, A1) / h
    C = torch.where(Co <= 0.5, Co * (1.0 - Co), torch.full_like(Co, 0.25))
    G = torch.where(flat, torch.zeros_like(C), 0.5 * C * (2.0 - phi(sp / safe) - phi(sm / safe)))
    Dn = G * d0
    if periodic:
        new = mean + Dn - down(Dn)
        return torch.cat([X[:, :1], new[:, 1:-1], X[:, -1:]], 1)
    Dn = Dn * h
    zero = torch.zeros_like(Dn[:, :1])
    inside = mean[:, 1:-1] + (torch.cat([Dn, zero], 1) - torch.cat([zero, Dn], 1)) / m.w[1:-1]
    return torch.cat([mean[:, :1], inside, mean[:, -1:]], 1)


def _cfl(m, X):
    u, T, _ = _primitives(m, X)
    c = torch.sqrt(m.cs2 * T)
    return 0.5 * min(float(((m.h_cfl if a == "z" else m.h[a]) / (u[a].abs() + c)).min()) for a in m.axes)


def _step(m, X, dt, mu=None, kth=None, frozen=False):
    for along in 2 * list(reversed(m.axes)):
        X = _sweep(m, X, along, 0.5 * dt, m.mu if mu is None else mu, m.kth if kth is None else kth, frozen)
    return X


def _volume(m, f):
    return float((f.mean((1, 2), keepdim=True) * m.w).sum())


def _plate_nu(m, X):
    """Mean of the two plates' Nusselt numbers: derivative of the quadratic through the three nearest planes."""
    f = (_primitives(m, X)[1] - (1.0 - m.D * m.z)).mean((1, 2))

    def slope(f0, f1, f2, h1, h2):
        return -(2 * h1 + h2) / (h1 * (h1 + h2)) * f0 + (h1 + h2) / (h1 * h2) * f1 - h1 / (h2 * (h1 + h2)) * f2

    z = m.planes
    bottom = slope(f[0], f[1], f[2], z[1] - z[0], z[2] - z[1])
    top = -slope(f[-1], f[-2], f[-3], z[-1] - z[-2], z[-2] - z[-3])
    return -(bottom + top) / (2.0 * EPS)


def _analysis(m, X):
    """Plane means of the z-momentum terms and of the profiles, C and max K_e/I_e."""
    u, T, p = _primitives(m, X)
    rho, nz = X[0], m.nz
    a, b = m.hp[:-1], m.hp[1:]

    def ddz(f):
        return -b / (a * (a + b)) * f[:-2] + (b - a) / (a * b) * f[1:-1] + a / (b * (a + b)) * f[2:]

    def ddx(f):
        return (torch.roll(f, -1, 2) - torch.roll(f, 1, 2)) / (2.0 * m.h["x"])

    ux, uz, inner = u["x"], u["z"], slice(1, -1)
    uxx = (torch.roll(uz, -1, 2) - 2.0 * uz + torch.roll(uz, 1, 2)) / m.h["x"] ** 2
    uzz = 2.0 * (uz[:-2] / (a * (a + b)) - uz[1:-1] / (a * b) + uz[2:] / (b * (a + b)))
    mean = lambda f: f.mean((1, 2))  # noqa: E731
    pad = lambda f: torch.nn.functional.pad(mean(f), (1, 1))  # noqa: E731
    Tsa, z = T - (1.0 - m.D * m.z), m.z[:, 0, 0]
    out = {"F_n": pad(rho[inner] * (ux * ddx(uz))[inner] + rho[inner] * uz[inner] * ddz(uz)), "F_p": pad(-ddz(p)),
           "F_b": pad(m.g * rho[inner]),
           "F_v": pad(m.mu * (uxx[inner] + (2.0 - 2.0 / 3.0) * uzz + (1.0 - 2.0 / 3.0) * ddz(ddx(ux)))),
           "rho_uz_sq": mean((rho * uz) ** 2), "Tsa_sq": mean(Tsa ** 2), "Tsa": mean(T) - (1.0 - m.D * z),
           "rho_minus_rhoA": mean(rho) - (1.0 - m.D * z) ** (1.0 / (m.gamma - 1.0)),
           "U": torch.sqrt(mean(ux * ux + uz * uz))}
    C = _volume(m, rho * uz * Tsa) / math.sqrt(_volume(m, (rho * uz) ** 2) * _volume(m, Tsa ** 2))
    r_max = float((0.5 * (ux * ux + uz * uz) * m.b / T).max())
    assert out["F_n"].numel() == nz
    return {"profiles": out, "hist": None, "C": C, "r_max": r_max}


def exact(case, seed):
    if case["kind"] == "batch":
        return None  # thousands of steps of many boxes take minutes with whole-array operations
    device = "cuda" if torch.cuda.is_available() else "cpu"
    m = _Model(case, device)
    if case["kind"] == "adjoint":
        from torch.utils.checkpoint import checkpoint
        X0 = _field(m, seed, torch.float64).requires_grad_()
        Ra = torch.tensor(case["Ra"], dtype=torch.float64, device=device, requires_grad=True)
        mu, kth = torch.sqrt(m.Pr / Ra), 1.0 / (EPS * m.D * torch.sqrt(Ra * m.Pr))
        X, J = X0, 0.0
        for s in range(1, case["steps"] + 1):
            dt = _cfl(m, X.detach())
            X = checkpoint(lambda Y, p, q, dt=dt: _step(m, Y, dt, p, q, True), X, mu, kth, use_reentrant=False)
            if s >= case["win"]:
                J = J + _plate_nu(m, X)
        J = J / (case["steps"] - case["win"] + 1)
        dX, dRa = torch.autograd.grad(J, (X0, Ra))
        return {"J": J.detach(), "dX": dX[:, :, 0].contiguous(), "dRa": dRa}
    dtype = torch.float64 if case["prec"] == "fp64" else torch.float32
    with torch.no_grad():
        X = _field(m, seed, dtype).double()
        if case["kind"] == "analysis":
            return _analysis(m, X)
        seen = []

        def sample():
            seen.append((_volume(m, X[-1]), _volume(m, 0.5 * (X[1:-1] ** 2).sum(0) / X[0])))

        for s in range(1, case["steps"] + 1):
            X = _step(m, X, m.fixed_dt() if case["via"] == "device" else _cfl(m, X))
            if case["diag_every"] and s % case["diag_every"] == 0:
                sample()
        if case["via"] == "host":
            sample()
            X = X if case["ndim"] == 3 else X[:, :, 0].contiguous()
        return {"X": X, "energy": [e for e, _ in seen], "KE": [k for _, k in seen]}
