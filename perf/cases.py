"""The workloads whose speed is measured: what programs have the evaluator do on the GPU.

An optimal control program builds a problem once and then, in every iteration of its solver, asks
for the objective, the constraints, their derivatives, products with them and the KKT values at
a new point.  The cases are such calls through the package's public entry points
(`ocp.OCP`, `ocp.OCPBatch`, `autograd`), from horizons of some tens of nodes, where a
call's latency counts, to a million nodes, for every model, both schemes and the options that
change the work (path and boundary inequalities, a boundary cost, a free final time, parameters on
the device, host buffers).  Everything is FP64: the evaluator has no other type.

`exact` restates the transcription in plain torch (node derivatives by torch.func).
"""
import math

import torch

from paper_2510_03932_gb300 import autograd, ocp

# ---- problems -------------------------------------------------------------------------------
# Model data: states, controls, parameters, horizon T, cost weights q and r, initial state, the
# ranges of the states and the control, and the sparsity of the dynamics: the state and control
# columns of each row's defect, and the lower pairs with a second derivative.
INF = float("inf")
MODELS = {
    "vdp": dict(nx=2, nu=1, p=[1.0], T=10.0, q=[1.0, 1.0], r=[1.0], x0=[1.0, 0.0], x=(-1.0, 1.0), u=(-1.0, 1.0),
                xv=[[0, 1], [0, 1]], uv=[[], [0]], hess=[(0, 0), (1, 0)]),
    "dint": dict(nx=2, nu=1, p=[], T=1.0, q=[0.0, 0.0], r=[0.5], x0=[-1.0, 0.0], xf=[0.0, 0.0], x=(-1.0, 1.0),
                 u=(-1.0, 1.0), xv=[[0, 1], [1]], uv=[[], [0]], hess=[]),
    "cartpole": dict(nx=4, nu=1, p=[1.0, 0.1, 0.5, 9.81], T=5.0, q=[1.0] * 4, r=[0.1], x0=[0.0] * 4, x=(-1.0, 1.0),
                     u=(-10.0, 10.0), xv=[[0, 1], [1, 2, 3], [2, 3], [2, 3]], uv=[[], [0], [], [0]],
                     hess=[(2, 2), (3, 2), (3, 3), (4, 2)]),
    "quadrotor": dict(nx=9, nu=4, p=[9.8], T=1.0, q=[0.5, 0.0, 0.5, 0.0, 0.5, 0.0, 0.5, 0.5, 0.5], r=[0.05] * 4,
                      x0=[0.0] * 9, x=(-1.0, 1.0), u=(-10.0, 10.0),
                      slope={4: 2.0}, sine={0: (1.0, 2 * math.pi), 2: (2.0, 4 * math.pi)},
                      xv=[[0, 1], [1, 6, 7, 8], [2, 3], [3, 6, 7, 8], [4, 5], [5, 6, 7], [6, 7], [6, 7], [6, 7, 8]],
                      uv=[[], [0], [], [0], [], [0], [1, 2], [1, 2], [1, 2, 3]],
                      hess=[(6, 6), (7, 6), (7, 7), (8, 6), (8, 7), (8, 8), (9, 6), (9, 7), (9, 8), (10, 6), (10, 7),
                            (11, 6), (11, 7)]),
    "goddard": dict(nx=3, nu=1, p=[310.0, 500.0, 3.5, 2.0], T=1.0, q=[0.0] * 3, r=[0.0], x0=[1.0, 0.0, 1.0], xf=[0.6],
                    xf_comp=[2], mayer=[-1.0, 0.0, 0.0], tf=(0.15, 0.25), x=[(1.0, 1.02), (0.0, 0.1), (0.6, 1.0)],
                    u=(0.0, 1.0), xv=[[0, 1], [0, 1, 2], [2]], uv=[[], [0], [0]],
                    hess=[(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2), (3, 2)]),
}
# FP64 operations of one node's evaluation (F, c, gradient, J and H) and of its three products,
# rounded: the models' formulas with every intermediate formed once.
OPS = {"vdp": (26, 36), "dint": (12, 24), "cartpole": (110, 250), "quadrotor": (235, 500), "goddard": (94, 220)}
# Path inequalities, rows of {variable: (a, b, l)} with right-hand side r (a half-space and control
# bounds, a box and an ellipse, an altitude band, a keep-out disc and a tilt bound, ...).
PATH = {
    "vdp": [({1: (0.0, 0.0, -1.0)}, 0.4), ({2: (1.0, 0.0, 0.0)}, 1.0)],
    "dint": [({2: (1.0, 0.0, 0.0)}, 4.0)],
    "cartpole": [({0: (0.25, 0.0, 0.0), 2: (1.0, 0.0, 0.0)}, 1.0), ({4: (1.0, 0.0, 0.0)}, 100.0)],
    "quadrotor": [({4: (1.0, 1.0, 0.0)}, 1.0), ({0: (-1.0, 0.5, 0.0), 2: (-1.0, 0.5, 0.0)}, -0.04),
                  ({6: (1.0, 0.0, 0.0), 7: (1.0, 0.0, 0.0)}, 0.5)],
    "goddard": [({1: (0.0, 0.0, 1.0)}, 0.1), ({3: (1.0, 0.0, 0.0)}, 1.0)],
}
# Boundary inequalities over (X_0, X_N): terminal sets and start-end couplings.
ENDS = {
    "vdp": [({2: (1.0, 0.0, 0.0), 3: (1.0, 0.0, 0.0)}, 0.25), ({0: (0.0, 0.0, -1.0), 2: (0.0, 0.0, 1.0)}, 1.0)],
    "dint": [({3: (1.0, 0.0, 0.0)}, 0.01)],
    "cartpole": [({6: (1.0, math.pi, 0.0)}, 0.01), ({0: (0.0, 0.0, -1.0), 4: (0.0, 0.0, 1.0)}, 0.5)],
    "quadrotor": [({9: (1.0, 1.0, 0.0), 11: (1.0, 1.0, 0.0)}, 0.1), ({4: (0.0, 0.0, 1.0), 13: (0.0, 0.0, -1.0)}, -1.0)],
    "goddard": [({0: (0.0, 0.0, 1.0), 3: (0.0, 0.0, -1.0)}, -1e-3), ({4: (1.0, 0.0, 0.0)}, 0.01)],
}


def _rows(rows, nz):
    d = dict(a=[], b=[], l=[], r=[])
    for terms, r in rows:
        for i, key in enumerate("abl"):
            d[key].append([terms.get(v, (0.0, 0.0, 0.0))[i] for v in range(nz)])
        d["r"].append(r)
    return d


def _problem(case, N=None, r=None, x0=None):
    """The case's problem as plain data (N, r, x0: one instance of a batch)."""
    name = case["model"]
    if name == "heat":
        n = case["cells"]
        P = dict(nx=n, nu=1, p=[float(n)], T=1.0, q=[1.0] * n, r=[1e-2], xref=[0.5] * n, x0=[0.0] * n, x=(0.0, 1.0),
                 u=(-1.0, 1.0), xv=[[v for v in (k - 1, k, k + 1) if 0 <= v < n] for k in range(n)],
                 uv=[[0] if k == 0 else [] for k in range(n)], hess=[(k, k) for k in range(n)])
    else:
        P = dict(MODELS[name])
    P.update(model=name, N=int(N or case["N"]), scheme=case.get("scheme", "trapezoid"))
    if r is not None:
        P.update(r=r, x0=x0)
    nx, nz = P["nx"], P["nx"] + P["nu"]
    P["path"] = _rows(PATH[name], nz) if case.get("path") else None
    P["bineq"] = P["bolza"] = None
    if case.get("ends"):
        P["bineq"] = _rows(ENDS[name], 2 * nx)
        a, b = [0.5] + [0.0] * (nx - 1) + [1.5] * nx, [0.0] * nx + [0.1 * (k + 1) for k in range(nx)]
        P["bolza"] = dict(a=a, b=b, l=[-0.25] + [0.0] * (2 * nx - 2) + [0.3])
    P["nun"] = P["N"] if P["scheme"] == "euler" else P["N"] + 1
    P["nfin"] = len(P.get("xf") or [])
    P["n"] = nx * (P["N"] + 1) + P["nu"] * P["nun"] + (1 if "tf" in P else 0)
    P["m"] = nx + P["nfin"] + nx * P["N"] + (len(P["path"]["r"]) * P["nun"] if P["path"] else 0) + \
        (len(P["bineq"]["r"]) if P["bineq"] else 0)
    return P


def _handle(P):
    nx, slope, sine = P["nx"], P.get("slope", {}), P.get("sine", {})
    track = (None, None, None)
    if slope or sine:
        track = ([slope.get(k, 0.0) for k in range(nx)], [sine.get(k, (0.0, 0.0))[0] for k in range(nx)],
                 [sine.get(k, (0.0, 0.0))[1] for k in range(nx)])
    return ocp.OCP(P["model"], nx, P["nu"], P["N"], P["T"], P["p"], P["q"], P["r"], P.get("xref"), None, P["x0"],
                   P.get("xf"), *track, free_tf="tf" in P, xf_comp=P.get("xf_comp"), mayer=P.get("mayer"),
                   scheme=P["scheme"], path=P["path"], bineq=P["bineq"], bolza=P["bolza"])


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, k, lo, hi):
    return torch.rand(k, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _normal(g, k):
    return torch.randn(k, generator=g, device="cuda", dtype=torch.float64)


def _point(P, g):
    """x: states and controls uniform over the model's operating range (and tf)."""
    nodes, nx = P["N"] + 1, P["nx"]
    if isinstance(P["x"], list):
        X = torch.stack([_uniform(g, nodes, lo, hi) for lo, hi in P["x"]], 1).reshape(-1)
    else:
        X = _uniform(g, nx * nodes, *P["x"])
    parts = [X, _uniform(g, P["nu"] * P["nun"], *P["u"])]
    if "tf" in P:
        parts.append(_uniform(g, 1, *P["tf"]))
    return torch.cat(parts)


# ---- cases ----------------------------------------------------------------------------------
def listed():
    return [
        # the smallest step of a control loop: four tiles, the call's latency
        dict(name="vdp step, N 1000", call="step", model="vdp", N=1000),
        # the headline benchmark: one fused step of the million-node Van der Pol problem
        dict(name="vdp step, N 1e6", call="step", model="vdp", N=1_000_000),
        # a solver's five callbacks, each in a call of its own
        dict(name="cartpole callbacks, N 1e5", call="callbacks", model="cartpole", N=100_000),
        # one interior-point iteration at the paper's largest quadrotor horizon: F, c, gradient, J, H, KKT
        dict(name="quadrotor iteration, N 1e5", call="iteration", model="quadrotor", N=100_000),
        # the same for the rocket with its free final time (a dense column of J and row of H)
        dict(name="goddard iteration, N 1e5", call="iteration", model="goddard", N=100_000),
        # the discretised heat equation's fused step
        dict(name="heat 64 step, N 2e4", call="step", model="heat", cells=64, N=20_000),
        # an iterative linear solver's products at a ragged size
        dict(name="heat 37 products, N 7003", call="products", model="heat", cells=37, N=7003),
        # many problems at once: 256 cart-poles with uneven horizons
        dict(name="cartpole batch of 256", call="batch", model="cartpole", count=256, nmin=500, nmax=50_000),
        # fitting parameters: c(x; p) and F(x) forward, their vector-Jacobian product backward
        dict(name="cartpole adjoint, N 1e6", call="adjoint", model="cartpole", N=1_000_000),
        # an iteration with path and boundary inequalities and a boundary cost, ragged horizon
        dict(name="constrained quadrotor, N 33333", call="iteration", model="quadrotor", N=33_333, path=True, ends=True),
        # forward Euler with path inequalities: the callbacks of a coarse first solve
        dict(name="euler cartpole, N 250001", call="callbacks", model="cartpole", N=250_001, scheme="euler", path=True),
        # a solver on the host: pinned arrays in and out, copies included
        dict(name="vdp host step, N 1e5", call="host", model="vdp", N=100_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["step", "step", "callbacks", "callbacks", "iteration", "iteration", "products", "adjoint", "batch", "host"])
    if call == "batch":
        nmin = _log(rng, 20, 2000)
        return dict(call=call, model=rng.choice(["vdp", "dint", "cartpole", "cartpole"]), count=_log(rng, 4, 256), nmin=nmin,
                    nmax=nmin + _log(rng, 10, 48_000))
    if call == "adjoint":
        return dict(call=call, model=rng.choice(["vdp", "cartpole", "quadrotor"]), N=_log(rng, 50, 300_000))
    if call == "host":
        return dict(call=call, model=rng.choice(["vdp", "dint"]), N=_log(rng, 50, 100_000))
    model = rng.choice(["vdp", "dint", "cartpole", "quadrotor", "goddard", "heat"])
    if model == "heat":
        cells = _log(rng, 2, 128)
        return dict(call=call, model=model, cells=cells, N=_log(rng, 50, min(100_000, 1_280_000 // cells)))
    most = {"vdp": 1_000_000, "dint": 1_000_000, "cartpole": 300_000, "quadrotor": 100_000, "goddard": 200_000}[model]
    case = dict(call=call, model=model, N=_log(rng, 50, most), path=rng.random() < 0.4)
    if model != "goddard" and rng.random() < 0.25:
        case["scheme"] = "euler"
    elif rng.random() < 0.4:
        case["ends"] = True
    return case


def _batch(case):
    """The instances of a batch: horizons, control weights and initial states, by a fixed sequence."""
    out, s = [], case["count"] * 2654435761 + case["nmax"]
    nx = MODELS[case["model"]]["nx"]
    for _ in range(case["count"]):
        u = []
        for _ in range(2 + nx):
            s = (s * 6364136223846793005 + 1442695040888963407) % 2**64
            u.append((s >> 33) / 2.0**31)
        N = case["nmin"] + int(u[0] * (case["nmax"] - case["nmin"] + 1))
        out.append(_problem(case, N=N, r=[0.01 + 0.99 * u[1]], x0=[v - 0.5 for v in u[2:]]))
    return out


def _data(case, seed):
    """The inputs of a case: the point x, multipliers y, directions vn and vm, sigma_x."""
    g = _gen(seed)
    if case["call"] == "batch":
        Ps = _batch(case)
        x = torch.cat([_point(P, g) for P in Ps])
        return Ps, dict(x=x, y=_normal(g, sum(P["m"] for P in Ps)))
    P = _problem(case)
    d = dict(x=_point(P, g), y=_normal(g, P["m"]), vn=_uniform(g, P["n"], -1.0, 1.0), vm=_normal(g, P["m"]))
    if case["call"] == "iteration":
        d["sx"] = _uniform(g, P["n"], 0.0, 10.0)
    if case["call"] == "adjoint":
        d["p"] = torch.tensor(P["p"], dtype=torch.float64, device="cuda") * _uniform(g, len(P["p"]), 0.9, 1.1)
        d["one"] = torch.ones((), dtype=torch.float64, device="cuda")
    return P, d


SIGMA, DELTA_W, DELTA_C = 1.0, 1e-4, 1e-8


def prepare(case, seed):
    P, d = _data(case, seed)
    s = dict(call=case["call"], **d)
    if case["call"] == "batch":
        s["H"] = ocp.OCPBatch([_handle(p) for p in P])
        s["outs"] = s["H"].outputs()
        return s
    H = s["H"] = _handle(P)
    e = lambda k: torch.empty(k, dtype=torch.float64, device="cuda")  # noqa: E731
    if case["call"] == "host":
        for k in ("x", "y", "vn", "vm"):
            s[k] = s[k].cpu().pin_memory()
        s["outs"] = [torch.empty(k, dtype=torch.float64).pin_memory() for k in (1, H.m, H.n, H.nnzj, H.nnzh, H.m, H.n, H.n)]
    elif case["call"] == "step":
        s["outs"] = [e(k) for k in (1, H.m, H.n, H.nnzj, H.nnzh, H.m, H.n, H.n)]
    elif case["call"] == "products":
        s["outs"] = [e(H.m), e(H.n), e(H.n)]
    elif case["call"] == "adjoint":
        s["x"].requires_grad_(True)
        s["p"].requires_grad_(True)
    else:
        s["outs"] = [e(k) for k in (1, H.m, H.n, H.nnzj, H.nnzh)]
        if case["call"] == "iteration":
            s["kkt"] = e(H.kkt_nnz())
    return s


def run(s):
    H, call = s["H"], s["call"]
    if call == "step":
        return H.eval_step(s["x"], s["y"], SIGMA, s["vn"], s["vm"], outs=s["outs"])
    if call == "host":
        return H.eval_step_host(s["x"], s["y"], SIGMA, s["vn"], s["vm"], outs=s["outs"])
    if call == "callbacks":
        f, c, g, jv, hv = s["outs"]
        H.eval_obj(s["x"], f)
        H.eval_cons(s["x"], c)
        H.eval_grad(s["x"], g)
        H.jac_coo_values(s["x"], jv)
        H.hess_coo_values(s["x"], s["y"], SIGMA, hv)
        return s["outs"]
    if call == "iteration":
        f, c, g, jv, hv = H.eval_all(s["x"], s["y"], SIGMA, *s["outs"])
        return f, c, g, jv, hv, H.kkt_values(hv, jv, s["sx"], DELTA_W, DELTA_C, out=s["kkt"])
    if call == "products":
        jv, jtv, hv = s["outs"]
        H.jprod(s["x"], s["vn"], jv)
        H.jtprod(s["x"], s["vm"], jtv)
        H.hprod(s["x"], s["y"], SIGMA, s["vn"], hv)
        return s["outs"]
    if call == "batch":
        H.eval_all(s["x"], s["y"], SIGMA, *s["outs"])
        return s["outs"]
    # adjoint: reverse-mode derivatives of c(x; p) and F(x)
    c = autograd.constraints(H, s["x"], s["p"])
    F = autograd.objective(H, s["x"])
    gx, gp = torch.autograd.grad((c, F), (s["x"], s["p"]), (s["vm"], s["one"]))
    return c.detach(), F.detach(), gx, gp


# ---- the work a pass cannot do without -------------------------------------------------------
def _hess_template(P):
    """The structural (a, b) pairs of a node's Hessian block, X rows then U rows, and all pairs."""
    nx, nz = P["nx"], P["nx"] + P["nu"]
    w = P["q"] + P["r"]
    pairs = set(P["hess"])
    for v in range(nz):
        sq = w[v] != 0.0
        if P["path"]:
            sq = sq or any(a[v] != 0.0 for a in P["path"]["a"])
        if P["bineq"] and v < nx:
            sq = sq or any(a[v] != 0.0 or a[nx + v] != 0.0 for a in P["bineq"]["a"] + [P["bolza"]["a"]])
        if sq:
            pairs.add((v, v))
    pairs = sorted(pairs)
    return [ab for ab in pairs if ab[0] < nx], [ab for ab in pairs if ab[0] >= nx]


def _counts(P):
    """(nnz of J, nnz of H, entries of the KKT matrix) of a problem."""
    nx, nu, N, nun, tf = P["nx"], P["nu"], P["N"], P["nun"], 1 if "tf" in P else 0
    nb = nx + P["nfin"]
    if P["scheme"] == "euler":
        per = sum(len(P["xv"][k]) + 1 + len(P["uv"][k]) for k in range(nx))
    else:
        per = sum(2 * (len(P["xv"][k]) + len(P["uv"][k])) + tf for k in range(nx))
    extra = 0
    if P["path"]:
        extra += nun * sum(a != 0.0 or b != 0.0 for ra, rl in zip(P["path"]["a"], P["path"]["l"]) for a, b in zip(ra, rl))
    if P["bineq"]:
        extra += sum(a != 0.0 or b != 0.0 for ra, rl in zip(P["bineq"]["a"], P["bineq"]["l"]) for a, b in zip(ra, rl))
    X, U = _hess_template(P)
    nnzj, nnzh = nb + per * N + extra, (len(X) + len(U)) * nun + 4 * tf * nun
    missing = nx + nu - sum(a == b for a, b in X + U)
    return nnzj, nnzh, nnzj + nnzh + P["m"] + missing * nun + (nx if P["scheme"] == "euler" else 0) + tf


def work(case):
    Ps = _batch(case) if case["call"] == "batch" else [_problem(case)]
    doubles, flops, call = 0, 0, case["call"]
    for P in Ps:
        n, m, nodes = P["n"], P["m"], P["N"] + 1
        nnzj, nnzh, nnzk = _counts(P)
        ev, pr = OPS.get(P["model"], (18 * P["nx"], 19 * P["nx"]))
        evaluated = 1 + m + n + nnzj + nnzh
        if call in ("step", "host"):
            doubles += 2 * n + 2 * m + evaluated + m + 2 * n
            flops += (ev + pr) * nodes
        elif call in ("callbacks", "batch"):
            doubles += n + m + evaluated
            flops += ev * nodes
        elif call == "iteration":
            doubles += n + m + evaluated + n + nnzk
            flops += ev * nodes
        elif call == "products":
            doubles += 2 * n + 2 * m + m + 2 * n
            flops += pr * nodes
        else:
            doubles += n + m + m + 1 + n + 2 * len(P["p"])
            flops += 2 * ev * nodes
    return {"bytes": 8 * doubles, "flops": flops}


# ---- the values in plain torch ---------------------------------------------------------------
def _f(model, z, p):
    """Dynamics of one node (z a vector)."""
    if model == "vdp":
        return torch.stack([z[1], p[0] * (1 - z[0] ** 2) * z[1] - z[0] + z[2]])
    if model == "dint":
        return torch.stack([z[1], z[2]])
    if model == "cartpole":
        mc, mp, l, g = p[0], p[1], p[2], p[3]
        s, c, w, F = torch.sin(z[2]), torch.cos(z[2]), z[3], z[4]
        D = mc + mp * s * s
        return torch.stack([z[1], (F + mp * s * (l * w * w + g * c)) / D, w,
                            (-F * c - mp * l * w * w * c * s - (mc + mp) * g * s) / (l * D)])
    if model == "quadrotor":
        u1, u2, u3, u4 = z[9], z[10], z[11], z[12]
        s7, c7, s8, c8, s9, c9 = torch.sin(z[6]), torch.cos(z[6]), torch.sin(z[7]), torch.cos(z[7]), torch.sin(z[8]), torch.cos(z[8])
        a = u2 * c7 + u3 * s7
        return torch.stack([z[1], u1 * (c7 * s8 * c9 + s7 * s9), z[3], u1 * (c7 * s8 * s9 - s7 * c9), z[5],
                            u1 * c7 * c8 - p[0], a / c8, u3 * c7 - u2 * s7, a * s8 / c8 + u4])
    r, v, m, u = z[0], z[1], z[2], z[3]  # goddard
    Cd, beta, Tmax, b = p[0], p[1], p[2], p[3]
    return torch.stack([v, -Cd * v * v * torch.exp(-beta * (r - 1)) / m - 1 / r**2 + u * Tmax / m, -b * Tmax * u])


def _derivs(P, z, yb, p):
    """f, its Jacobian and sum_k yb_k Hess f_k at every node (rows of z)."""
    if P["model"] == "heat":
        n = P["nx"]
        x, u, i2 = z[:, :n], z[:, n:], float(n) ** 2
        left, right = torch.cat([u, x[:, :-1]], 1), torch.cat([x[:, 1:], x[:, -1:]], 1)
        f = (left - 2 * x + right) * i2 - x**3
        J, H = z.new_zeros(z.shape[0], n, n + 1), z.new_zeros(z.shape[0], n + 1, n + 1)
        k = torch.arange(n, device=z.device)
        J[:, k, k] = -2 * i2 - 3 * x**2
        J[:, n - 1, n - 1] += i2
        J[:, k[1:], k[1:] - 1] = i2
        J[:, k[:-1], k[:-1] + 1] = i2
        J[:, 0, n] = i2
        H[:, k, k] = -6 * x * yb
        return f, J, H
    fn = lambda zz: _f(P["model"], zz, p)  # noqa: E731
    out = ([], [], [])
    for zc, yc in zip(z.split(200_000), yb.split(200_000)):
        out[0].append(torch.func.vmap(fn)(zc))
        out[1].append(torch.func.vmap(torch.func.jacfwd(fn))(zc))
        out[2].append(torch.func.vmap(torch.func.jacfwd(torch.func.jacrev(lambda zz, yy: (yy * fn(zz)).sum())))(zc, yc))
    return tuple(torch.cat(o) for o in out)


def _reference(P, d, x, y):
    """Every output of the problem at (x, y) as a dict (products where d has directions)."""
    nx, nu, N, nun, euler = P["nx"], P["nu"], P["N"], P["nun"], P["scheme"] == "euler"
    h = (x[-1] / N) if "tf" in P else torch.tensor(P["T"] / N, dtype=torch.float64, device=x.device)
    s = h if euler else h / 2                 # the step on one node's dynamics
    nX = nx * (N + 1)

    def nodes(v):  # (nun, nz): the entries of v on the nodes that have a control
        return torch.cat([v[:nX].reshape(N + 1, nx)[:nun], v[nX:nX + nu * nun].reshape(nun, nu)], 1)

    nb = nx + P["nfin"]

    def bar(w):    # defect multipliers summed over the rows of each node
        r = w[nb:nb + nx * N].reshape(nx, N).T
        return r if euler else torch.cat([r, r.new_zeros(1, nx)]) + torch.cat([r.new_zeros(1, nx), r])

    z, X, yb = nodes(x), x[:nX].reshape(N + 1, nx), bar(y)
    pars = d["p"].detach() if "p" in d else torch.tensor(P["p"], dtype=torch.float64, device=x.device)
    f, Jf, Hf = _derivs(P, z, yb, pars)
    D = -s * Jf                               # the node's share of its rows, identity excluded
    # objective, gradient, and the Hessian of the running cost
    wq = torch.full((nun,), 1.0, dtype=torch.float64, device=x.device)
    if not euler:
        wq[0] = wq[-1] = 0.5
    wq = (wq * h)[:, None] * torch.tensor(P["q"] + P["r"], dtype=torch.float64, device=x.device)
    ref = torch.tensor((P.get("xref") or [0.0] * nx) + [0.0] * nu, dtype=torch.float64, device=x.device).repeat(nun, 1)
    t = torch.arange(nun, dtype=torch.float64, device=x.device) * h
    for k, v in P.get("slope", {}).items():
        ref[:, k] += v * t
    for k, (amp, freq) in P.get("sine", {}).items():
        ref[:, k] += amp * torch.sin(freq * t)
    F = (wq * (z - ref) ** 2).sum()
    gz = 2 * wq * (z - ref)
    Hn = SIGMA * torch.diag_embed(2 * wq) - s * Hf
    if "mayer" in P:
        mayer = torch.tensor(P["mayer"], dtype=torch.float64, device=x.device)
        F = F + (mayer * X[-1]).sum()
    gX = x.new_zeros(N + 1, nx)
    gX[:nun] = gz[:, :nx]
    if "mayer" in P:
        gX[-1] += mayer
    # constraint rows
    fin = (P.get("xf_comp") or list(range(nx))) if P["nfin"] else []
    fr = f if euler else f[:-1] + f[1:]
    c = [X[0], X[-1][fin], (X[1:] - X[:-1] - s * fr).T.reshape(-1)]
    ji = [x.new_ones(nb)]
    eye = torch.eye(nx, nx + nu, dtype=torch.float64, device=x.device)
    L = D - eye if euler else D[:-1] - eye
    R = None if euler else D[1:] + eye
    for k in range(nx):
        xv, uv = P["xv"][k], [nx + i for i in P["uv"][k]]
        if euler:
            rows = [L[:, k, xv], x.new_ones(N, 1), L[:, k, uv]]
        else:
            rows = [L[:, k, xv], R[:, k, xv], L[:, k, uv], R[:, k, uv]]
        if "tf" in P:
            rows.append(-fr[:, k:k + 1] / (2 * N))
        ji.append(torch.cat(rows, 1).reshape(-1))
    # path inequalities, boundary inequalities and the boundary cost
    yp = y[nb + nx * N:]
    paths, ends = [], []
    if P["path"]:
        for p, r in enumerate(P["path"]["r"]):
            a, b, l = (torch.tensor(P["path"][k][p], dtype=torch.float64, device=x.device) for k in "abl")
            dz = 2 * a * (z - b) + l
            c.append((a * (z - b) ** 2 + l * z).sum(1) - r)
            ji.append(dz[:, (a != 0) | (l != 0)].reshape(-1))
            Hn = Hn + torch.diag_embed(2 * a * yp[p * nun:(p + 1) * nun, None])
            paths.append(dz)
        yp = yp[len(paths) * nun:]
    if P["bineq"]:
        ze = torch.cat([X[0], X[-1]])
        He = x.new_zeros(2 * nx)
        for q, r in enumerate(P["bineq"]["r"]):
            a, b, l = (torch.tensor(P["bineq"][k][q], dtype=torch.float64, device=x.device) for k in "abl")
            dz = 2 * a * (ze - b) + l
            c.append(((a * (ze - b) ** 2 + l * ze).sum() - r).reshape(1))
            ji.append(dz[(a != 0) | (l != 0)])
            He = He + 2 * a * yp[q]
            ends.append(dz)
        a, b, l = (torch.tensor(P["bolza"][k], dtype=torch.float64, device=x.device) for k in "abl")
        F = F + (a * (ze - b) ** 2 + l * ze).sum()
        gX[0] += (2 * a * (ze - b) + l)[:nx]
        gX[-1] += (2 * a * (ze - b) + l)[nx:]
        He = He + SIGMA * 2 * a
        k = torch.arange(nx, device=x.device)
        Hn[0, k, k] += He[:nx]
        Hn[-1, k, k] += He[nx:]
    tail = [x.new_zeros(1)] if "tf" in P else []
    HX, HU = _hess_template(P)
    pick = lambda t: torch.stack([Hn[:, a, b] for a, b in t], 1).reshape(-1) if t else x.new_zeros(0)  # noqa: E731
    hi = [pick(HX), pick(HU)]
    if "tf" in P:
        tr = -(yb[:, :, None] * Jf).sum(1) / (2 * N)          # the tf row on every node's variables
        hi += [tr[:, :nx].reshape(-1), tr[:, nx:].reshape(-1)]
    out = dict(f=F.reshape(1), c=torch.cat(c), g=torch.cat([gX.reshape(-1), gz[:, nx:].reshape(-1)] + tail), j=torch.cat(ji),
               h=torch.cat(hi))
    if "sx" in d:   # KKT values: rows of the (1, 1) block, then the constraint rows, each with its diagonal last
        sx, k = d["sx"], []
        sz = nodes(sx)
        for lo, hi_ in ((0, nx), (nx, nx + nu)):
            cols = []
            for a in range(lo, hi_):
                bs = [b for aa, b in HX + HU if aa == a]
                cols += [Hn[:, a, b] + (sz[:, a] + DELTA_W if a == b else 0.0) for b in bs]
                if a not in bs:
                    cols.append(sz[:, a] + DELTA_W)
            k.append(torch.stack(cols, 1).reshape(-1))
            if euler and lo == 0:
                k.append(sx[nx * N:nX] + DELTA_W)
        if "tf" in P:
            k += [hi[2], hi[3], sx[-1:] + DELTA_W]
        k.append(torch.stack([ji[0], torch.full_like(ji[0], -DELTA_C)], 1).reshape(-1))
        sizes = [N] * nx + [nun] * len(paths) + [1] * len(ends)
        for row, rows in zip(ji[1:], sizes):
            e = row.reshape(rows, -1)
            k.append(torch.cat([e, torch.full_like(e[:, :1], -DELTA_C)], 1).reshape(-1))
        out["k"] = torch.cat(k)
    if "vn" not in d:
        return out
    # products
    v, w = d["vn"], d["vm"]
    vz, vX, wb, wr = nodes(v), v[:nX].reshape(N + 1, nx), bar(w), w[nb:nb + nx * N].reshape(nx, N)
    pv = (D * vz[:, None, :]).sum(2)
    rows = (pv if euler else pv[:-1] + pv[1:]) + vX[1:] - vX[:-1]
    if "tf" in P:
        rows = rows - fr / (2 * N) * v[-1]
    Jv = [vX[0], vX[-1][fin], rows.T.reshape(-1)]
    o = (D * wb[:, :, None]).sum(1)
    oX = x.new_zeros(N + 1, nx)
    oX[:nun] += o[:, :nx]
    oX[1:] += wr.T
    oX[:-1] -= wr.T
    oX[0] += w[:nx]
    if fin:
        oX[-1, fin] += w[nx:nb]
    oU, wp = o[:, nx:].clone(), w[nb + nx * N:]
    for p, dz in enumerate(paths):
        Jv.append((dz * vz).sum(1))
        oX[:nun] += (wp[p * nun:(p + 1) * nun, None] * dz)[:, :nx]
        oU += (wp[p * nun:(p + 1) * nun, None] * dz)[:, nx:]
    wp = wp[len(paths) * nun:]
    for q, dz in enumerate(ends):
        Jv.append((dz * torch.cat([vX[0], vX[-1]])).sum().reshape(1))
        oX[0] += wp[q] * dz[:nx]
        oX[-1] += wp[q] * dz[nx:]
    Hs = torch.tril(Hn) + torch.tril(Hn, -1).transpose(1, 2)
    Hv = (Hs * vz[:, None, :]).sum(2)
    jt, ht = [], []
    if "tf" in P:
        Hv = Hv + tr * v[-1]
        jt, ht = [-(wr.T * fr).sum().reshape(1) / (2 * N)], [(tr * vz).sum().reshape(1)]
    HvX = x.new_zeros(N + 1, nx)
    HvX[:nun] = Hv[:, :nx]
    out.update(jv=torch.cat(Jv), jt=torch.cat([oX.reshape(-1), oU.reshape(-1)] + jt),
               hv=torch.cat([HvX.reshape(-1), Hv[:, nx:].reshape(-1)] + ht))
    if "p" in d:
        pp = pars.clone().requires_grad_(True)
        fp = torch.func.vmap(lambda zz: _f(P["model"], zz, pp))(z)
        out["dp"] = torch.autograd.grad((-s * wb * fp).sum(), pp)[0]
    return out


def exact(case, seed):
    P, d = _data(case, seed)
    if case["call"] == "batch":
        parts, xo, yo = [], 0, 0
        for p in P:
            parts.append(_reference(p, {}, d["x"][xo:xo + p["n"]], d["y"][yo:yo + p["m"]]))
            xo, yo = xo + p["n"], yo + p["m"]
        return [torch.cat([o[k] for o in parts]) for k in ("f", "c", "g", "j", "h")]
    o = _reference(P, d, d["x"], d["y"])
    if case["call"] == "adjoint":
        return o["c"], o["f"].reshape(()), o["jt"] + o["g"], o["dp"]
    keys = {"step": "f c g j h jv jt hv", "host": "f c g j h jv jt hv", "callbacks": "f c g j h", "iteration": "f c g j h k",
            "products": "jv jt hv"}[case["call"]]
    out = [o[k] for k in keys.split()]
    return [t.cpu() for t in out] if case["call"] == "host" else out
