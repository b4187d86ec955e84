"""The work that users of the library have it do, as cases that can be timed and compared.

Every case is one problem of the kinds the library solves (Besse & Xing's Schwarz waveform
relaxation on (a0, b0) x (0, T)), at the sizes of the benchmark workloads
(paper_1503_02564_gb300/workloads.py, bench.py) and of the smoke check:

  solve   V(x): swr_build_interface + swr_solve (GMRES with the causal preconditioner), the
          scaling workload's step, with Robin or S_0^2 transmission
  build   V(x): swr_build_interface and the interface problem copied out (d, first columns)
  batch   many uneven V(x) instances in one plan
  time    V(t,x): matrix-free GMRES with the mean-potential preconditioner
  nonlin  |u|^2 + V0(x): preconditioned fixed point, misfit and gradient
  adjoint V(x): solve, misfit and gradient
  apply   one application of the interface operator R on a built plan
  algebra (I - L) x and the preconditioner on a built plan

The plan is what a user's program keeps from call to call; a pass takes the inputs (potential
and initial value, or an interface vector) through the public entry points.
"""
import math

import numpy as np
import torch

from paper_1503_02564_gb300 import swr

P_ROBIN = complex(math.sqrt(5.0) * np.exp(-1j * math.pi / 4))


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: the smoke check's problem, bound by launches and latency
        {"name": "solve_tiny", "kind": "solve", "nx": 241, "h": 0.1, "nt": 30, "nsub": 4, "dt": 1e-3, "tc": 0},
        # the plain workload: 1001 nodes, four subdomains
        {"name": "solve_plain", "kind": "solve", "nx": 1001, "h": 0.024, "nt": 200, "nsub": 4, "dt": 1e-3, "tc": 0},
        # the scaling workload with few long subdomains (12501 nodes each)
        {"name": "solve_n16", "kind": "solve", "nx": 200001, "h": 5e-4, "nt": 500, "nsub": 16, "dt": 1e-3, "tc": 0},
        # the scaling workload with many short subdomains (401 nodes each)
        {"name": "solve_n500", "kind": "solve", "nx": 200001, "h": 5e-4, "nt": 500, "nsub": 500, "dt": 1e-3, "tc": 0},
        # the order-2 transmission condition S_0^2 (end histories) on a ragged partition
        {"name": "solve_s02_n61", "kind": "solve", "nx": 100003, "h": 5e-4, "nt": 300, "nsub": 61, "dt": 1e-3, "tc": 1},
        # the interface problem alone, kept by a program that solves it itself
        {"name": "build_n256", "kind": "build", "nx": 200001, "h": 5e-4, "nt": 500, "nsub": 256, "dt": 1e-3, "tc": 0},
        # 48 independent instances of uneven sizes and step counts in one plan
        {"name": "batch_48", "kind": "batch", "count": 48, "h": 1e-3, "dt": 1e-3, "sub_lo": 200, "sub_hi": 2000,
         "n_lo": 4, "n_hi": 64, "nx_hi": 40000, "nt_lo": 100, "nt_hi": 400, "mix": 1},
        # a moving well: one march of all subdomains per Krylov iteration
        {"name": "time_n64", "kind": "time", "nx": 60001, "h": 1e-3, "nt": 400, "nsub": 64, "dt": 1e-3},
        # the cubic nonlinearity: forward solve, misfit and gradient
        {"name": "nonlin_n32", "kind": "nonlin", "nx": 20001, "h": 2e-3, "nt": 400, "nsub": 32, "dt": 5e-4},
        # the gradient of a linear problem, checkpointed every 50 steps
        {"name": "adjoint_n64", "kind": "adjoint", "nx": 200001, "h": 5e-4, "nt": 500, "nsub": 64, "dt": 1e-3, "ckpt": 50},
        # one application of R (a program's own outer iteration, the classical algorithm)
        {"name": "apply_n256", "kind": "apply", "nx": 200001, "h": 5e-4, "nt": 500, "nsub": 256, "dt": 1e-3, "tc": 0},
        # the interface algebra of a Krylov method that the program runs itself
        {"name": "algebra_n500", "kind": "algebra", "nx": 200001, "h": 5e-4, "nt": 500, "nsub": 500, "dt": 1e-3, "tc": 0},
    ]


def _log(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def draw(rng):
    """Problems of the ranges above: 241 to 200001 nodes, 30 to 500 steps, 2 to 500 subdomains
    of at least 0.2 (the width the preconditioners are made for), Robin and S_0^2."""
    kind = rng.choice(["solve", "solve", "solve", "build", "batch", "time", "nonlin", "adjoint", "apply", "algebra"])
    if kind == "batch":
        lo = int(_log(rng, 200, 500))
        return {"kind": kind, "count": int(_log(rng, 4, 48)), "h": 1e-3, "dt": 1e-3, "sub_lo": lo,
                "sub_hi": int(lo * (2 + 2 * rng.random())), "n_lo": 4, "n_hi": rng.randint(8, 40),
                "nx_hi": 40000, "nt_lo": rng.randint(50, 150), "nt_hi": rng.randint(160, 400), "mix": rng.randint(2, 1 << 20)}
    if kind == "time":
        nx = int(_log(rng, 3000, 60001))
        nsub = max(2, min(64, int(_log(rng, 2, nx / 400))))
        return {"kind": kind, "nx": nx, "h": 1e-3, "nt": int(_log(rng, 40, 300)), "nsub": nsub, "dt": 1e-3}
    if kind == "nonlin":
        nx = int(_log(rng, 1500, 20001))
        nsub = max(2, min(32, int(_log(rng, 2, nx / 200))))
        return {"kind": kind, "nx": nx, "h": 2e-3, "nt": int(_log(rng, 40, 400)), "nsub": nsub, "dt": 5e-4}
    if kind == "solve" and rng.random() < 0.35:
        nx = int(_log(rng, 241, 4001))
        return {"kind": kind, "nx": nx, "h": 24.0 / (nx - 1), "nt": int(_log(rng, 30, 500)),
                "nsub": rng.randint(2, 8), "dt": 1e-3, "tc": rng.randint(0, 1)}
    nx = int(_log(rng, 5000, 200001))
    nsub = max(2, min(500, int(_log(rng, 2, nx / 400))))
    if kind == "adjoint":
        nsub = max(nsub, nx // 20000 + 2)
        return {"kind": kind, "nx": nx, "h": 5e-4, "nt": int(_log(rng, 50, 400)), "nsub": nsub, "dt": 1e-3,
                "ckpt": rng.choice([20, 50, 0])}
    return {"kind": kind, "nx": nx, "h": 5e-4, "nt": int(_log(rng, 50, 500)), "nsub": nsub, "dt": 1e-3,
            "tc": rng.randint(0, 1) if kind != "algebra" else 0}


# --------------------------------------------------------------------------
# inputs: wells and packets, drawn from the seed
# --------------------------------------------------------------------------
def _dev():
    return torch.device("cuda:0")


def _offsets(nx, nsub):
    base, extra = divmod(nx - 1, nsub)
    sizes = np.full(nsub, base, dtype=np.int64)
    sizes[:extra] += 1
    return np.concatenate([[0], np.cumsum(sizes)])


def _grid(case):
    half = 0.5 * (case["nx"] - 1) * case["h"]
    return np.linspace(-half, half, case["nx"])


def _packets(x, rng, count, width):
    span = 0.3 * (x[-1] - x[0])
    u = np.zeros_like(x, dtype=np.complex128)
    for _ in range(count):
        c, w, k, ph = rng.uniform(-span, span), rng.uniform(*width), rng.uniform(-10, 10), rng.uniform(0, 2 * math.pi)
        u += np.exp(-(x - c) ** 2 / (2 * w * w) + 1j * (k * x + ph))
    return u


def _static_inputs(case, rng):
    """A sum of wells (or the inverted oscillator of the plain workload) and wave packets."""
    x = _grid(case)
    if case["nx"] <= 4001 and case["kind"] == "solve":
        V = -x * x / 4 * rng.uniform(0.8, 1.2)
        u0 = np.exp(-((x - rng.uniform(-1, 1)) ** 2) / 2 + 5j * x) * np.exp(1j * rng.uniform(-1e-3, 1e-3, x.size))
        return V, u0
    V = np.zeros_like(x)
    span = 0.4 * (x[-1] - x[0])
    for _ in range(8):
        V -= 5.0 * np.exp(-(x - rng.uniform(-span, span)) ** 2 / (2 * rng.uniform(0.5, 3.0) ** 2))
    return V, _packets(x, rng, 4, (0.5, 2.0))


def _batch_inputs(case, rng):
    """Grids, partitions and step counts belong to the case; potentials and states to the seed."""
    mix, out = np.random.default_rng(case["mix"]), []
    for _ in range(case["count"]):
        while True:
            n = int(mix.integers(case["n_lo"], case["n_hi"] + 1))
            el = mix.integers(case["sub_lo"] - 1, case["sub_hi"], size=n)
            nx = int(el.sum()) + 1
            if nx <= case["nx_hi"]:
                break
        half = 0.5 * (nx - 1) * case["h"]
        x = -half + case["h"] * np.arange(nx)
        V = np.zeros(nx)
        for _ in range(4):
            V += rng.uniform(-10, 10) * np.exp(-(x - rng.uniform(-half, half)) ** 2 / (2 * rng.uniform(0.5, 3.0) ** 2))
        out.append({"nx": nx, "a0": -half, "b0": half, "nt": int(mix.integers(case["nt_lo"], case["nt_hi"] + 1)),
                    "nsub": n, "node_off": np.concatenate([[0], np.cumsum(el)]), "V": V, "u0": _packets(x, rng, 1, (0.5, 2.0))})
    return out


def _time_inputs(case, rng):
    x = torch.tensor(_grid(case), dtype=torch.float64, device=_dev())
    amp, om = rng.uniform(4.0, 6.0), rng.uniform(0.8, 1.2)
    t = (torch.arange(case["nt"] + 1, dtype=torch.float64, device=_dev()) * case["dt"])[:, None]
    V = -x * x / 4 * (1 + 0.5 * torch.sin(4 * t)) - 10 * torch.exp(-((x - amp * torch.sin(om * t)) ** 2))
    x0, k0 = rng.uniform(-0.15, 0.15) * float(x[-1] - x[0]), rng.uniform(-5, 5)
    u0 = torch.exp(torch.complex(-((x - x0) ** 2) / 2, k0 * x))
    return V.contiguous(), u0


def _nonlin_inputs(case, rng):
    x = _grid(case)
    span = 0.375 * (x[-1] - x[0])
    V, Vt = np.zeros_like(x), np.zeros_like(x)
    for _ in range(6):
        d, c, w = rng.uniform(2, 10), rng.uniform(-span, span), rng.uniform(0.5, 2.0)
        b = np.exp(-((x - c) ** 2) / (2 * w * w))
        V -= d * b
        Vt -= d * (1 + 0.05 * rng.standard_normal()) * b
    u0 = np.exp(2j * x) / np.cosh(x - rng.uniform(-0.5, 0.5))
    # the target: the initial state with a phase that the perturbed wells would give it
    tgt = u0 * np.exp(1j * Vt * case["nt"] * case["dt"])
    return V, u0, tgt


def _random_interface(n, rng):
    return rng.standard_normal(n) + 1j * rng.standard_normal(n)


def prepare(case, seed):
    rng = np.random.default_rng([20150309, int(seed)])
    dev, kind = _dev(), case["kind"]
    c = lambda a: torch.tensor(a, dtype=torch.complex128, device=dev)  # noqa: E731
    f = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
    s = {"kind": kind}
    if kind == "batch":
        ins = _batch_inputs(case, rng)
        s["plan"] = swr.BatchPlan(ins, dt=case["dt"], p=P_ROBIN, restart=30, maxit=2000, tol_abs=1e-10,
                                  precond=swr.SWR_PC_CAUSAL)
        s["V"] = f(np.concatenate([i["V"] for i in ins]))
        s["u0"] = c(np.concatenate([i["u0"] for i in ins]))
    else:
        off = _offsets(case["nx"], case["nsub"])
        half = 0.5 * (case["nx"] - 1) * case["h"]
        common = dict(nx=case["nx"], a0=-half, b0=half, nt=case["nt"], dt=case["dt"], nsub=case["nsub"],
                      node_off=off, p=P_ROBIN, tol_abs=1e-10)
        if kind == "time":
            s["V"], s["u0"] = _time_inputs(case, rng)
            s["V"] = s["V"].view(-1)
            s["plan"] = swr.Plan(vkind=swr.SWR_V_TIME, restart=60, maxit=400,
                                 precond=swr.SWR_PC_MEAN_POTENTIAL, **common)
        elif kind == "nonlin":
            V, u0, tgt = _nonlin_inputs(case, rng)
            s["V"], s["u0"], s["target"] = f(V), c(u0), c(tgt)
            s["plan"] = swr.Plan(vkind=swr.SWR_V_NONLINEAR, solver=swr.SWR_SOLVER_FIXED_POINT, maxit=200,
                                 precond=swr.SWR_PC_MEAN_POTENTIAL, nl_tol=1e-13, nl_maxit=50, **common)
        else:
            V, u0 = _static_inputs(case, rng)
            s["V"], s["u0"] = f(V), c(u0)
            s["plan"] = swr.Plan(tc=case.get("tc", 0), restart=30, maxit=2000, precond=swr.SWR_PC_CAUSAL, **common)
            if kind == "adjoint":
                noise = _random_interface(case["nx"], rng)
                s["target"] = c(u0 * np.exp(0.4j) + 0.05 * noise)
    plan = s["plan"]
    e = lambda n: torch.empty(n, dtype=torch.complex128, device=dev)  # noqa: E731
    if kind in ("apply", "algebra"):   # the program has built the interface problem
        s["x"] = c(_random_interface(plan.n_interface, rng))
        s["y"], s["z"] = e(plan.n_interface), e(plan.n_interface)
        plan.build_interface(s["V"], s["u0"])
    elif kind == "build":
        s["d"], s["cols"] = e(plan.n_interface), e(plan.n_cols)
    else:
        s["g"], s["uT"] = e(plan.n_interface), e(plan.nx)
        if kind in ("nonlin", "adjoint"):
            s["ubar"] = e(plan.nx)
            s["grad"] = torch.empty(plan.nx, dtype=torch.float64, device=dev)
            s["ckpt"] = case.get("ckpt", 0)
    return s


def run(s):
    plan, kind = s["plan"], s["kind"]
    if kind == "apply":
        plan.apply_R(s["x"], s["y"])
        return {"Rg": s["y"]}
    if kind == "algebra":
        plan.apply_interface(s["x"], s["y"])
        plan.apply_precond(s["y"], s["z"])
        return {"y": s["y"], "z": s["z"]}
    plan.build_interface(s["V"], s["u0"])
    if kind == "build":
        plan.get_interface(s["d"], s["cols"])
        return {"d": s["d"], "cols": s["cols"]}
    plan.solve(s["g"], False, s["uT"])
    if kind in ("nonlin", "adjoint"):
        J = plan.misfit(s["uT"], s["target"], s["ubar"])
        plan.adjoint(s["ubar"], s["grad"], s["ckpt"])
        return {"g": s["g"], "uT": s["uT"], "J": J, "grad": s["grad"]}
    return {"g": s["g"], "uT": s["uT"]}


def work(case):
    """36 flops per node, step and march (a tridiagonal solve with stored factors); the marches a
    method cannot do without: both unit impulses and the zero-flux march per subdomain (V(x)),
    one march of the grid per outer iteration otherwise (taken as 12 for the nonlinear fixed
    point and 40 for GMRES with V(t,x)); inputs once, outputs once."""
    kind = case["kind"]
    if kind == "batch":
        nx = case["count"] * 0.25 * (case["n_lo"] + case["n_hi"]) * (case["sub_lo"] + case["sub_hi"])
        nx = min(nx, case["count"] * case["nx_hi"])
        nt = 0.5 * (case["nt_lo"] + case["nt_hi"])
        ni = case["count"] * (case["n_lo"] + case["n_hi"]) * nt
        return {"flops": 36.0 * 3 * nx * nt, "bytes": 24.0 * nx + 16.0 * (nx + ni)}
    nx, nt, n = case["nx"], case["nt"], case["nsub"]
    ni = (2.0 * n - 2) * nt
    marches = {"solve": 3, "build": 3, "adjoint": 6, "time": 40, "nonlin": 14, "apply": 1, "algebra": 0}[kind]
    flops = 36.0 * marches * nx * nt
    nbytes = 24.0 * nx + 16.0 * (nx + ni)
    if kind == "algebra":
        lg = math.log2(max(2, 2 * nt))
        flops = 2.0 * ni * 2 * (2 * 5 * lg)       # two applies by fast convolution
        nbytes = 16.0 * (4 * n * nt + 3 * ni)
    elif kind == "build":
        nbytes = 24.0 * nx + 16.0 * (4 * n * nt + ni)
    elif kind == "apply":
        nbytes = 16.0 * (nx + 2 * ni)
    elif kind == "time":
        nbytes += 8.0 * nx * nt
    elif kind in ("nonlin", "adjoint"):
        nbytes += 16.0 * nx + 8.0 * nx
    return {"flops": flops, "bytes": nbytes}


# --------------------------------------------------------------------------
# the same outputs from a plain march of the whole grid (or of each subdomain) in torch:
# P1 elements, Crank-Nicolson, the tridiagonal systems by cyclic reduction over whole vectors
# --------------------------------------------------------------------------
def _matrices(V, h, dt):
    """Diagonal and coupling of A = (2i/dt) M - S + M_V on the last axis' grid."""
    z = torch.zeros_like(V[..., :1])
    el = torch.ones_like(V[..., 1:])
    left, right = torch.cat([z, el], -1), torch.cat([el, z], -1)      # elements at each node
    lo, hi = torch.cat([z, V[..., :-1] + 3 * V[..., 1:]], -1), torch.cat([3 * V[..., :-1] + V[..., 1:], z], -1)
    d = torch.complex(-(left + right) / h + h / 12 * (lo + hi), 2 / dt * h / 3 * (left + right))
    e = torch.complex(1 / h + h / 12 * (V[..., :-1] + V[..., 1:]), torch.full_like(el, 2 / dt * h / 6))
    return d, e


class _Tri:
    """Cyclic reduction of a symmetric tridiagonal matrix on the last axis (batched)."""

    def __init__(self, d, e):
        n = d.shape[-1]
        lo = torch.cat([torch.zeros_like(d[..., :1]), e], -1)
        up = torch.cat([e, torch.zeros_like(d[..., :1])], -1)
        self.levels, st = [], 1
        while st < n:
            a, g = -lo[..., st:] / d[..., :-st], -up[..., :-st] / d[..., st:]
            nd = d.clone()
            nd[..., st:] += a * up[..., :-st]
            nd[..., :-st] += g * lo[..., st:]
            nl, nu = torch.zeros_like(lo), torch.zeros_like(up)
            nl[..., st:] = a * lo[..., :-st]
            nu[..., :-st] = g * up[..., st:]
            self.levels.append((st, a, g))
            lo, up, d, st = nl, nu, nd, 2 * st
        self.inv = 1 / d

    def solve(self, r):
        for st, a, g in self.levels:
            o = r.clone()
            o[..., st:].addcmul_(a, r[..., :-st])
            o[..., :-st].addcmul_(g, r[..., st:])
            r = o
        return r * self.inv


def _mass(u, h):
    r = u.clone()
    r[..., 1:-1] *= 2
    r = r * (h / 3)
    r[..., 1:] += h / 6 * u[..., :-1]
    r[..., :-1] += h / 6 * u[..., 1:]
    return r


def _beta(n, dev):
    b = torch.zeros(n + 2, dtype=torch.float64, device=dev)
    a = 1.0
    for k in range(0, n + 1, 2):
        b[k], b[k + 1] = a, -a
        a *= (k + 1) / (k + 2)
    return b[: n + 1]


def _sbar(v, tc, dt):
    """The transmission operator on traces v[..., 0..nt] (v_0 = u_0), entries 1..nt."""
    if tc == 0:
        return P_ROBIN * v[..., 1:]
    n = v.shape[-1] - 1
    c2 = complex(np.exp(-0.25j * math.pi) * math.sqrt(2 / dt))
    m = 4 * (n + 1)
    y = torch.fft.ifft(torch.fft.fft(_beta(n, v.device).to(torch.complex128), m) * torch.fft.fft(v, m, dim=-1), dim=-1)
    return c2 * y[..., 1:n + 1]


def _form(x, y, h):
    """Re x^T (dM_W / dW_k) y for every node k."""
    s = (x * y).real
    c = (x[..., :-1] * y[..., 1:] + x[..., 1:] * y[..., :-1]).real
    r = torch.zeros_like(s)
    r[..., :-1] += h / 12 * (3 * s[..., :-1] + c + s[..., 1:])
    r[..., 1:] += h / 12 * (s[..., :-1] + c + 3 * s[..., 1:])
    return r


def _interface(vs, us, Ws, off_count, h, dt, tc):
    """g from the whole grid's solution near the interfaces: vs[K, 3, nt+1], us likewise,
    Ws[K, 3, nt] or [K, 3, 1] the potential that step n saw."""
    I2 = 2j / dt
    vm, v0, vp = vs[:, 0, 1:], vs[:, 1, 1:], vs[:, 2, 1:]
    um, u0, up = us[:, 0, :-1], us[:, 1, :-1], us[:, 2, :-1]
    Wm, W0, Wp = Ws[:, 0], Ws[:, 1], Ws[:, 2]
    dnl = (I2 * (h / 6 * (um - vm) + h / 3 * (u0 - v0)) + (v0 - vm) / h
           - (h / 12 * (Wm + W0) * vm + h / 12 * (Wm + 3 * W0) * v0))
    dnr = (I2 * (h / 3 * (u0 - v0) + h / 6 * (up - vp)) + (v0 - vp) / h
           - (h / 12 * (3 * W0 + Wp) * v0 + h / 12 * (W0 + Wp) * vp))
    sv = _sbar(vs[:, 1], tc, dt)
    return torch.stack([dnl + sv, dnr + sv], 1).reshape(-1)   # r_j, l_{j+1} of every interface


def _near(off, dev):
    k = torch.tensor(np.asarray(off[1:-1]), device=dev)
    return torch.stack([k - 1, k, k + 1], 1)


def _exact_static(case, s, adjoint=False):
    V, u, h, dt, nt = s["V"], s["u0"], case["h"], case["dt"], case["nt"]
    dev, off = V.device, _offsets(case["nx"], case["nsub"])
    I2 = 2j / dt
    d, e = _matrices(V, h, dt)
    tri, at = _Tri(d, e), _near(off, dev)
    vs = torch.zeros(at.shape + (nt + 1,), dtype=torch.complex128, device=dev)
    us = torch.zeros_like(vs)
    vs[..., 0] = us[..., 0] = u[at]
    every = []
    for n in range(1, nt + 1):
        v = tri.solve(I2 * _mass(u, h))
        u = 2 * v - u
        vs[..., n], us[..., n] = v[at], u[at]
        if adjoint:
            every.append(v)
    g = _interface(vs, us, V[at][..., None], None, h, dt, case.get("tc", 0))
    out = {"g": g, "uT": u}
    if adjoint:
        err = u - s["target"]
        out["J"] = float((err.conj() * _mass(err, h)).sum().real)
        z = (2 * err).conj() * (dt / 2j)
        grad = torch.zeros_like(V)
        for n in range(nt, 0, -1):
            w = tri.solve(I2 * _mass(z, h))
            grad -= 2 * _form(w, every[n - 1], h)
            z = 2 * w - z
        out["grad"] = grad
    return out


def _exact_batch(case, rng):
    ins, dev = _batch_inputs(case, rng), _dev()
    n, h, dt = max(i["nx"] for i in ins), case["h"], case["dt"]
    I2 = 2j / dt
    D = torch.ones(len(ins), n, dtype=torch.complex128, device=dev)
    E = torch.zeros(len(ins), n - 1, dtype=torch.complex128, device=dev)
    u = torch.zeros_like(D)
    wd = torch.zeros(len(ins), n, dtype=torch.float64, device=dev)
    wo = torch.zeros(len(ins), n - 1, dtype=torch.float64, device=dev)
    for k, i in enumerate(ins):
        m = i["nx"]
        D[k, :m], E[k, :m - 1] = _matrices(torch.tensor(i["V"], device=dev), h, dt)
        u[k, :m] = torch.tensor(i["u0"], device=dev)
        wd[k, :m], wo[k, :m - 1] = 2 * h / 3, h / 6
        wd[k, 0] = wd[k, m - 1] = h / 3
    tri = _Tri(D, E)
    row = torch.cat([torch.full((3 * (i["nsub"] - 1),), k) for k, i in enumerate(ins)]).to(dev)
    col = torch.cat([_near(i["node_off"], dev).reshape(-1) for i in ins])
    top = max(i["nt"] for i in ins)
    vs = torch.zeros(row.numel(), top + 1, dtype=torch.complex128, device=dev)
    us = torch.zeros_like(vs)
    vs[:, 0] = us[:, 0] = u[row, col]
    last = [None] * len(ins)
    for t in range(1, top + 1):
        r = wd * u
        r[:, 1:] += wo * u[:, :-1]
        r[:, :-1] += wo * u[:, 1:]
        v = tri.solve(I2 * r)
        u = 2 * v - u
        vs[:, t], us[:, t] = v[row, col], u[row, col]
        for k, i in enumerate(ins):
            if i["nt"] == t:
                last[k] = u[k, :i["nx"]].clone()
    g, at = [], 0
    for i in ins:
        m = 3 * (i["nsub"] - 1)
        a = vs[at:at + m].reshape(-1, 3, top + 1)[..., :i["nt"] + 1]
        b = us[at:at + m].reshape(-1, 3, top + 1)[..., :i["nt"] + 1]
        W = torch.tensor(i["V"], device=dev)[_near(i["node_off"], dev)][..., None]
        g.append(_interface(a, b, W, None, h, dt, 0))
        at += m
    return {"g": torch.cat(g), "uT": torch.cat(last)}


def _exact_time(case, s):
    h, dt, nt = case["h"], case["dt"], case["nt"]
    V, u = s["V"].view(nt + 1, -1), s["u0"]
    at = _near(_offsets(case["nx"], case["nsub"]), V.device)
    vs = torch.zeros(at.shape + (nt + 1,), dtype=torch.complex128, device=V.device)
    us = torch.zeros_like(vs)
    Ws = torch.zeros(at.shape + (nt,), dtype=torch.float64, device=V.device)
    vs[..., 0] = us[..., 0] = u[at]
    for n in range(1, nt + 1):
        W = 0.5 * (V[n] + V[n - 1])
        v = _Tri(*_matrices(W, h, dt)).solve(2j / dt * _mass(u, h))
        u = 2 * v - u
        vs[..., n], us[..., n], Ws[..., n - 1] = v[at], u[at], W[at]
    return {"g": _interface(vs, us, Ws, None, h, dt, 0), "uT": u}


def _weighted(W, v, h):
    """M_W v with the P1 rule for the potential."""
    wd = torch.zeros_like(W)
    wd[..., 1:] += h / 12 * (W[..., :-1] + 3 * W[..., 1:])
    wd[..., :-1] += h / 12 * (3 * W[..., :-1] + W[..., 1:])
    wo = h / 12 * (W[..., :-1] + W[..., 1:])
    r = wd * v
    r[..., 1:] += wo * v[..., :-1]
    r[..., :-1] += wo * v[..., 1:]
    return r


def _exact_nonlin(case, s):
    h, dt, nt, V, u = case["h"], case["dt"], case["nt"], s["V"], s["u0"]
    I2 = 2j / dt
    at = _near(_offsets(case["nx"], case["nsub"]), V.device)
    tri = _Tri(*_matrices(V, h, dt))
    vs = torch.zeros(at.shape + (nt + 1,), dtype=torch.complex128, device=V.device)
    us = torch.zeros_like(vs)
    Ws = torch.zeros(at.shape + (nt,), dtype=torch.float64, device=V.device)
    vs[..., 0] = us[..., 0] = u[at]
    every, v = [], u

    def settle(step, x):
        for k in range(60):   # the inner fixed point contracts by about 1e-3 per iteration
            y = step(x)
            if k >= 4 and float((y - x).abs().max()) <= 1e-15 * float(y.abs().max()):
                return y
            x = y
        return x

    for n in range(1, nt + 1):
        b = I2 * _mass(u, h)
        v = settle(lambda z: tri.solve(b - _weighted(z.abs() ** 2, z, h)), v)
        u = 2 * v - u
        vs[..., n], us[..., n], Ws[..., n - 1] = v[at], u[at], (V + v.abs() ** 2)[at]
        every.append(v)
    out = {"g": _interface(vs, us, Ws, None, h, dt, 0), "uT": u}
    err = u - s["target"]
    out["J"] = float((err.conj() * _mass(err, h)).sum().real)
    z = (2 * err).conj() * (dt / 2j)
    grad, w = torch.zeros_like(V), torch.zeros_like(u)
    for n in range(nt, 0, -1):
        v = every[n - 1]
        b = I2 * _mass(z, h)
        w = settle(lambda y: tri.solve(b - _weighted(v.abs() ** 2, y, h) - 2 * v.conj() * _form(v, y, h)), w)
        grad -= 2 * _form(w, v, h)
        z = 2 * w - z
    out["grad"] = grad
    return out


class _Subdomains:
    """All subdomains of a V(x) problem as one batch of marches (padded to the longest)."""

    def __init__(self, case, V):
        self.h, self.dt, self.nt, self.tc = case["h"], case["dt"], case["nt"], case.get("tc", 0)
        off = _offsets(case["nx"], case["nsub"])
        self.N, dev = case["nsub"], V.device
        n = int(np.max(np.diff(off))) + 1
        self.n = torch.tensor(np.diff(off) + 1, device=dev)
        D = torch.ones(self.N, n, dtype=torch.complex128, device=dev)
        E = torch.zeros(self.N, n - 1, dtype=torch.complex128, device=dev)
        self.wd = torch.zeros(self.N, n, dtype=torch.float64, device=dev)
        self.wo = torch.zeros(self.N, n - 1, dtype=torch.float64, device=dev)
        self.ends = (torch.zeros(self.N, dtype=torch.long, device=dev), self.n - 1)
        c2 = complex(np.exp(-0.25j * math.pi) * math.sqrt(2 / self.dt))
        sig = P_ROBIN if self.tc == 0 else c2
        for j in range(self.N):
            a, m = int(off[j]), int(off[j + 1] - off[j]) + 1
            D[j, :m], E[j, :m - 1] = _matrices(V[a:a + m], self.h, self.dt)
            self.wd[j, :m], self.wo[j, :m - 1] = 2 * self.h / 3, self.h / 6
            self.wd[j, 0] = self.wd[j, m - 1] = self.h / 3
            if j > 0:
                D[j, 0] -= sig
            if j < self.N - 1:
                D[j, m - 1] -= sig
        self.off, self.tri, self.c2 = off, _Tri(D, E), c2

    def march(self, u0, g):
        """New fluxes from u0 (nodal, or None) and the flux blocks g[2N-2, nt]."""
        N, nt, dev = self.N, self.nt, self.wd.device
        u = torch.zeros_like(self.tri.inv)
        if u0 is not None:
            for j in range(N):
                m = int(self.n[j])
                u[j, :m] = u0[int(self.off[j]):int(self.off[j]) + m]
        k = torch.arange(N, device=dev)
        lin = torch.zeros(2, N, nt, dtype=torch.complex128, device=dev)
        lin[1, :-1], lin[0, 1:] = g[0::2], g[1::2]
        tr = torch.zeros(2, N, nt + 1, dtype=torch.complex128, device=dev)
        for e in (0, 1):
            tr[e, :, 0] = u[k, self.ends[e]]
        beta = _beta(nt, dev).to(torch.complex128)
        on = torch.ones(2, N, 1, device=dev)
        on[0, 0] = on[1, -1] = 0
        for t in range(1, nt + 1):
            r = self.wd * u
            r[:, 1:] += self.wo * u[:, :-1]
            r[:, :-1] += self.wo * u[:, 1:]
            r = (2j / self.dt) * r
            for e in (0, 1):
                add = -lin[e, :, t - 1]
                if self.tc:
                    add = add + self.c2 * on[e, :, 0] * (tr[e, :, :t] * beta[1:t + 1].flip(0)).sum(-1)
                r[k, self.ends[e]] += add
            v = self.tri.solve(r)
            u = 2 * v - u
            for e in (0, 1):
                tr[e, :, t] = v[k, self.ends[e]]
        out = torch.zeros_like(g)
        sv = 2 * _sbar(tr, self.tc, self.dt)
        out[0::2] = (sv[0] - lin[0])[1:]
        out[1::2] = (sv[1] - lin[1])[:-1]
        return out

    def columns(self):
        """First columns of the Toeplitz blocks: unit impulses at the left ends, then the right."""
        cols = torch.zeros(self.N, 4, self.nt, dtype=torch.complex128, device=self.wd.device)
        for which in (0, 1):
            g = torch.zeros(2 * self.N - 2, self.nt, dtype=torch.complex128, device=self.wd.device)
            g[(1, 0)[which]::2, 0] = 1
            o = self.march(None, g)
            hit = slice(1, None) if which == 0 else slice(None, -1)   # subdomains that were driven
            a = torch.zeros_like(cols[:, 0])
            b = torch.zeros_like(a)
            a[1:], b[:-1] = o[0::2], o[1::2]
            cols[hit, 0 + which], cols[hit, 2 + which] = a[hit], b[hit]
        return cols


def _conv(c, x):
    m = 2 * c.shape[-1]
    return torch.fft.ifft(torch.fft.fft(c, m) * torch.fft.fft(x, m))[..., : c.shape[-1]]


def exact(case, seed):
    kind, rng = case["kind"], np.random.default_rng([20150309, int(seed)])
    if kind == "batch":
        return _exact_batch(case, rng)
    dev = _dev()
    s = {}
    c = lambda a: torch.tensor(a, dtype=torch.complex128, device=dev)  # noqa: E731
    if kind == "time":
        s["V"], s["u0"] = _time_inputs(case, rng)
        return _exact_time(case, s)
    if kind == "nonlin":
        V, u0, tgt = _nonlin_inputs(case, rng)
        s = {"V": torch.tensor(V, device=dev), "u0": c(u0), "target": c(tgt)}
        return _exact_nonlin(case, s)
    V, u0 = _static_inputs(case, rng)
    s = {"V": torch.tensor(V, device=dev), "u0": c(u0)}
    if kind == "adjoint":
        s["target"] = c(u0 * np.exp(0.4j) + 0.05 * _random_interface(case["nx"], rng))
        return _exact_static(case, s, adjoint=True)
    if kind == "solve":
        return _exact_static(case, s)
    sub = _Subdomains(case, s["V"])
    ni = (2 * case["nsub"] - 2) * case["nt"]
    if kind == "build":
        d = sub.march(s["u0"], torch.zeros(2 * case["nsub"] - 2, case["nt"], dtype=torch.complex128, device=dev))
        return {"d": d.reshape(-1), "cols": sub.columns().reshape(-1)}
    x = c(_random_interface(ni, rng)).view(-1, case["nt"])
    if kind == "apply":
        return {"Rg": sub.march(s["u0"], x).reshape(-1)}
    cols = sub.columns()
    y = x.clone()
    xl, xr = torch.zeros(2, case["nsub"], case["nt"], dtype=torch.complex128, device=dev)
    xl[1:], xr[:-1] = x[1::2], x[0::2]
    y[0::2] -= (_conv(cols[:, 0], xl) + _conv(cols[:, 1], xr))[1:]
    y[1::2] -= (_conv(cols[:, 2], xl) + _conv(cols[:, 3], xr))[:-1]
    return {"y": y.reshape(-1), "z": x.reshape(-1)}
