"""The work that programs of this framework have it do, as measurable cases.

A pass goes through the public classes (``Solver``, ``BatchSolver``).  The sizes are those of
the repository's workloads (Taylor--Green vortex 32^3 p = 3 and p = 4, isentropic vortex 4^3
p = 3, viscous shock 25^3, shock tube 128 x 1 x 1, batches of 4^3..12^3 instances of p = 2..5)
and ragged meshes like those of its tests.  Every initial state is a closed form with seeded
noise (amplitude 1e-3, as in the noisy Taylor--Green workload) and a seeded origin.

``exact`` evaluates the same scheme in plain torch FP64 (none of the package's code): the
SBP-SAT right-hand side, the Runge--Kutta step and the per-element relaxation roots.
"""
import math

import numpy as np
import torch

from paper_2003_08831_gb300 import _binding as B
from paper_2003_08831_gb300.solver import BatchSolver, Solver

GAMMA = 1.4
PRECISIONS = {"fp64": B.ES_FP64, "mixed": B.ES_MIXED, "fp64x": B.ES_FP64X, "mixed_ff": B.ES_MIXED_FF}
RKS = {"bs3": B.ES_RK_BS3, "rk4": B.ES_RK_RK4, "rk65": B.ES_RK_RK65}
STAGES = {"bs3": 3, "rk4": 4, "rk65": 6}
SHOCK = (2.5, 10.0, 0.75, -1.0)  # Mach, Reynolds, Prandtl, frame speed of the viscous shock
SOD = ((1.0, 1.0), (0.125, 0.1))  # (rho, p) left and right
MAX_NODE_STAGES = 4.0e6 * 3       # a drawn single-instance pass is no larger than the largest listed one


def _case(name, op, flow, p, n, precision="fp64", steps=1, mu=0.0, diss=1, rk="bs3"):
    return {"name": name, "op": op, "flow": flow, "p": p, "nx": n[0], "ny": n[1], "nz": n[2],
            "precision": precision, "steps": steps, "mu": mu, "diss": diss, "rk": rk}


def listed():
    return [
        # one right-hand side with entropy rates on the smallest mesh: a caller with its own
        # time integrator (or a test harness); latency and launches
        _case("rhs_vortex_p3_4", "rhs", "vortex", 3, (4, 4, 4)),
        # the paper's convergence set-up, isentropic vortex: 20 steps on 4^3 elements
        _case("advance_vortex_p3_4", "advance", "vortex", 3, (4, 4, 4), steps=20),
        # a shock tube at the paper's resolution, RK(4,4), prescribed end states
        _case("advance_sod_p3_128", "advance", "sod", 3, (128, 1, 1), steps=10, rk="rk4"),
        # relaxation alone (a caller's own integrator hands in u_old, u_new, d_eta), ragged mesh
        _case("relax_step_p2_17x13x19", "relax_step", "tgv", 2, (17, 13, 19)),
        # one step with both sides of the local entropy inequality returned: six-stage method,
        # matrix dissipation, highest degree, ragged mesh
        _case("estimate_p5_11x9x13", "estimate", "tgv", 5, (11, 9, 13), diss=2, rk="rk65"),
        # many independent vortices of mixed degrees and sizes advanced together, states read back
        {"name": "batch_fp64_16", "op": "batch", "flow": "vortex", "count": 16, "nmax": 8, "steps": 10,
         "precision": "fp64", "rk": "bs3", "diss": 1, "mu": 0.0},
        # the moving viscous shock, Navier--Stokes with Dirichlet-penalty faces, RK(4,4)
        _case("advance_shock_p3_25", "advance", "shock", 3, (25, 25, 25), mu=1.0 / SHOCK[1], rk="rk4"),
        # production size, Euler Taylor--Green: FP64, float-float fluxes, mixed with float-float estimates
        _case("euler_tgv_fp64_p3_32", "advance", "tgv", 3, (32, 32, 32), steps=2),
        _case("euler_tgv_fp64x_p3_32", "advance", "tgv", 3, (32, 32, 32), "fp64x", steps=2),
        _case("euler_tgv_mixed_ff_p3_32", "advance", "tgv", 3, (32, 32, 32), "mixed_ff", steps=4),
        # production size, Navier--Stokes Taylor--Green: FP64, and mixed with FP64 estimates
        _case("ns_tgv_fp64_p4_32", "advance", "tgv", 4, (32, 32, 32), mu=1.0 / 1600.0),
        _case("ns_tgv_mixed_p4_32", "advance", "tgv", 4, (32, 32, 32), "mixed", mu=1.0 / 1600.0),
    ]


def draw(rng):
    op = rng.choice(["rhs", "advance", "advance", "advance", "advance", "estimate", "relax_step", "batch"])
    precision = rng.choice(["fp64", "fp64", "fp64", "mixed", "mixed_ff", "fp64x"])
    rk = rng.choice(["bs3", "bs3", "rk4", "rk65"])
    if op == "batch":
        return {"op": "batch", "flow": "vortex", "count": rng.randint(3, 24), "nmax": rng.randint(5, 8),
                "steps": rng.randint(2, 8), "precision": precision, "rk": rk, "diss": rng.choice([0, 1, 1, 2]), "mu": 0.0}
    p = rng.randint(2, 5)
    flow = rng.choice(["vortex", "tgv", "tgv", "shock", "sod"]) if op == "advance" else rng.choice(["vortex", "tgv"])
    if flow == "sod":
        n = (int(round(math.exp(rng.uniform(math.log(16), math.log(256))))), 1, 1)
        rk = "rk4" if rk == "bs3" else rk
    else:
        side = math.exp(rng.uniform(math.log(3.0), math.log(30.0)))
        n = tuple(max(2, int(round(side * rng.uniform(0.75, 1.33)))) for _ in range(3))
    mu = {"shock": 1.0 / SHOCK[1], "tgv": rng.choice([0.0, 1.0 / 1600.0])}.get(flow, 0.0)
    if op == "relax_step":
        mu, rk, precision = 0.0, "bs3", "fp64"
    steps = rng.randint(1, 4) if op == "advance" else 1

    def cost():
        return n[0] * n[1] * n[2] * (p + 1) ** 3 * STAGES[rk] * steps * (1.0 if mu == 0.0 else 2.0)
    while cost() > MAX_NODE_STAGES:
        if steps > 1:
            steps -= 1
        else:
            n = tuple(max(2, int(v * 0.85)) for v in n)
    c = _case("", op, flow, p, n, precision, steps, mu, rng.choice([0, 1, 1, 2]) if flow in ("vortex", "tgv") else 1, rk)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------
# inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _lgl(p):
    """LGL nodes and weights on [-1, 1] and the derivative matrix (Legendre closed forms)."""
    leg = np.polynomial.legendre.Legendre.basis(p)
    x = np.concatenate([[-1.0], np.sort(np.real(leg.deriv().roots())), [1.0]])
    for _ in range(4):  # polish the interior roots of P_p'
        x[1:-1] -= leg.deriv()(x[1:-1]) / leg.deriv(2)(x[1:-1])
    x = 0.5 * (x - x[::-1])
    v = leg(x)
    w = 2.0 / (p * (p + 1) * v * v)
    d = np.zeros((p + 1, p + 1))
    for i in range(p + 1):
        for j in range(p + 1):
            if i != j:
                d[i, j] = v[i] / (v[j] * (x[i] - x[j]))
    d[0, 0], d[p, p] = -p * (p + 1) / 4.0, p * (p + 1) / 4.0
    return x, w, d


class _Mesh:
    """Sizes, box and tables of a case's mesh; states have shape (5, nz, ny, nx, k, j, i)."""

    def __init__(self, flow, p, n):
        self.p, self.P1, self.n = p, p + 1, tuple(n)
        if flow == "tgv":
            self.lo, self.hi = (0.0,) * 3, (2.0 * math.pi,) * 3
        elif flow == "vortex":
            self.lo, self.hi = (0.0,) * 3, (10.0,) * 3
        elif flow == "shock":
            self.lo, self.hi = (-0.5,) * 3, (0.5,) * 3
        else:
            h = 0.5 / n[0]
            self.lo, self.hi = (0.0, -h, -h), (1.0, h, h)
        self.h = [(self.hi[m] - self.lo[m]) / n[m] for m in range(3)]
        self.K, self.Np = n[0] * n[1] * n[2], (p + 1) ** 3
        self.shape = (n[2], n[1], n[0], p + 1, p + 1, p + 1)
        self.x, self.w, self.D = _lgl(p)
        w = torch.tensor(self.w, device=_device())
        self.mass = w[:, None, None] * w[None, :, None] * w[None, None, :] * (self.h[0] * self.h[1] * self.h[2] / 8.0)

    def coords(self):
        out = []
        x = torch.tensor(self.x, device=_device())
        for m in range(3):
            e = torch.arange(self.n[m], device=_device(), dtype=torch.float64)
            c = self.lo[m] + self.h[m] * (e[:, None] + 0.5 * (1.0 + x[None, :]))
            view = [1] * 6
            view[2 - m], view[5 - m] = self.n[m], self.P1
            out.append(c.reshape(view).expand(self.shape))
        return out


def _conserved(rho, v, pr):
    ke = 0.5 * rho * sum(a * a for a in v)
    return torch.stack([rho] + [rho * a for a in v] + [pr / (GAMMA - 1.0) + ke])


def _shock_constants():
    mach, re, pr, speed = SHOCK
    vf = (2.0 + (GAMMA - 1.0) * mach ** 2) / ((GAMMA + 1.0) * mach ** 2)
    alpha = 2.0 * GAMMA / (GAMMA + 1.0) / (re * pr)
    enthalpy = 1.0 / (GAMMA - 1.0) / mach ** 2 + 0.5
    return vf, alpha, enthalpy, speed


def _shock_state(x, t):
    """The viscous shock (mass flux 1, constant total enthalpy) at position x and time t."""
    vf, alpha, enthalpy, speed = _shock_constants()
    c = (1.0 + vf) / (1.0 - vf)
    xi = x - speed * t
    lo, hi = torch.full_like(xi, vf), torch.ones_like(xi)
    for _ in range(80):
        mid = 0.5 * (lo + hi)
        at = 0.5 * alpha * (torch.log((1.0 - mid) * (mid - vf)) + c * torch.log((1.0 - mid) / (mid - vf)))
        lo, hi = torch.where(at > xi, mid, lo), torch.where(at > xi, hi, mid)
    u = 0.5 * (lo + hi)
    rho = 1.0 / u
    z = torch.zeros_like(u)
    return rho, [u + speed, z, z], (GAMMA - 1.0) / GAMMA * rho * (enthalpy - 0.5 * u * u)


def _state(flow, mesh, seed):
    """Closed-form initial state with seeded origin and noise, (5, nz, ny, nx, k, j, i)."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=_device())
    gen.manual_seed(int(rng.integers(1 << 62)))
    x, y, z = mesh.coords()
    if flow == "tgv":
        a, b, c = rng.uniform(0.0, 2.0 * math.pi, 3)
        x, y, z = x + a, y + b, z + c
        p0 = 1.0 / (GAMMA * 0.1 ** 2)
        v = [torch.sin(x) * torch.cos(y) * torch.cos(z), -torch.cos(x) * torch.sin(y) * torch.cos(z), torch.zeros_like(x)]
        pr = p0 + (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0) / 16.0
        rho = pr / p0
    elif flow == "vortex":
        centre, eps, mach = rng.uniform(0.0, 10.0, 2), rng.uniform(3.0, 6.0), rng.uniform(0.1, 0.5)
        dx = torch.remainder(x - centre[0] + 5.0, 10.0) - 5.0
        dy = torch.remainder(y - centre[1] + 5.0, 10.0) - 5.0
        g = 1.0 - (dx * dx + dy * dy)
        temp = 1.0 - eps * eps * mach * mach * (GAMMA - 1.0) / (8.0 * math.pi ** 2) * torch.exp(g)
        rho = temp ** (1.0 / (GAMMA - 1.0))
        e = eps / (2.0 * math.pi) * torch.exp(0.5 * g)
        v = [math.sqrt(0.5) - e * dy, math.sqrt(0.5) + e * dx, torch.zeros_like(x)]
        pr = rho * temp / (GAMMA * mach * mach)
    elif flow == "shock":
        rho, v, pr = _shock_state(x + 0.1 * rng.uniform(-1.0, 1.0), 0.0)
    else:
        s = 0.5 * (1.0 - torch.tanh((x - 0.5 + 0.02 * rng.uniform(-1.0, 1.0)) / 0.03))
        rho = SOD[1][0] + (SOD[0][0] - SOD[1][0]) * s
        pr = SOD[1][1] + (SOD[0][1] - SOD[1][1]) * s
        v = [torch.zeros_like(x) for _ in range(3)]
    r = [1e-3 * (2.0 * torch.rand(mesh.shape, generator=gen, device=_device(), dtype=torch.float64) - 1.0) for _ in range(4)]
    return _conserved(rho * (1.0 + r[0]), [v[k] + r[k + 1] for k in range(3)], pr)


def _dt(q, mesh, mu):
    """Fixed step from the initial state, Courant number 0.5 (and its viscous limit)."""
    v = q[1:4] / q[0]
    pr = (GAMMA - 1.0) * (q[4] - 0.5 * q[0] * (v * v).sum(0))
    c = torch.sqrt(GAMMA * pr / q[0])
    lam = float(sum((v[m].abs() + c) / mesh.h[m] for m in range(3)).max())
    dt = 0.5 / ((2 * mesh.p + 1) * lam)
    if mu > 0.0:
        k2 = sum(((2 * mesh.p + 1) / h) ** 2 for h in mesh.h)
        dt = min(dt, 0.5 * float(q[0].min()) / (mu * GAMMA / 0.72 * k2))
    return dt


def _sod_ends():
    out = []
    for rho, pr in SOD:
        out += [rho, 0.0, 0.0, 0.0, pr / (GAMMA - 1.0)]
    return out


def _instances(case, seed):
    """Sizes of a batch belong to the case; the vortices in them to the seed."""
    rng = np.random.default_rng(case["count"] * 1000 + case["nmax"])
    out = []
    for i in range(case["count"]):
        n = int(rng.integers(4, case["nmax"] + 1))
        mesh = _Mesh("vortex", int(rng.integers(2, 6)), (n, n, n))
        q = _state("vortex", mesh, seed * 1000 + i)
        out.append((mesh, q, _dt(q, mesh, 0.0)))
    return out


def _relax_inputs(case, seed):
    """u_old, u_new and the entropy change for which every element's root is near 1."""
    mesh = _Mesh(case["flow"], case["p"], (case["nx"], case["ny"], case["nz"]))
    u = _state(case["flow"], mesh, seed)
    d = _Reference(mesh, case).rhs(u, 0.0) * _dt(u, mesh, 0.0)
    gen = torch.Generator(device=_device())
    gen.manual_seed(seed + 7)
    g = 1.0 + 1e-3 * (2.0 * torch.rand(mesh.shape[:3], generator=gen, device=_device(), dtype=torch.float64) - 1.0)
    gd = g[..., None, None, None] * d
    deta = (_breg(u, gd, mesh)[0] + mesh_sum(mesh, (_entropy_vars(u) * gd).sum(0))) / g
    return mesh, u, u + d, deta


def prepare(case, seed):
    if case["op"] == "batch":
        inst = _instances(case, seed)
        b = BatchSolver([{"p": m.p, "n": m.n, "lo": m.lo, "hi": m.hi} for m, _, _ in inst],
                        precision=PRECISIONS[case["precision"]], rk=RKS[case["rk"]], interface_diss=case["diss"])
        for i, (_, q, _) in enumerate(inst):
            b.set_state(i, q.cpu().numpy())
        b.set_dt([dt for _, _, dt in inst])
        b.autotune()
        return {"case": case, "batch": b, "count": len(inst)}
    n = (case["nx"], case["ny"], case["nz"])
    mesh = _Mesh(case["flow"], case["p"], n)
    s = Solver(case["p"], n, mesh.lo, mesh.hi, mu=case["mu"], Pr=SHOCK[2] if case["flow"] == "shock" else 0.72,
               interface_diss=case["diss"], rk=RKS[case["rk"]], precision=PRECISIONS[case["precision"]])
    if case["flow"] == "shock":
        s.set_boundary(0, B.ES_BC_VISCOUS_SHOCK, SHOCK)
    elif case["flow"] == "sod":
        s.set_boundary(0, B.ES_BC_STATE, _sod_ends())
    state = {"case": case, "solver": s}
    if case["op"] == "relax_step":
        _, u, u_new, deta = _relax_inputs(case, seed)
        state.update(u=u.reshape(5, s.K, s.Np), u_new=u_new.reshape(5, s.K, s.Np), deta=deta.reshape(-1).contiguous())
        return state
    q = _state(case["flow"], mesh, seed)
    state["dt"] = _dt(q, mesh, case["mu"])
    state["q"] = q.reshape(5, s.K, s.Np).contiguous()
    if case["op"] != "rhs":
        s.autotune(state["q"])
    return state


def run(state):
    op = state["case"]["op"]
    if op == "batch":
        b = state["batch"]
        b.advance(state["case"]["steps"])
        t, gamma = b.times()
        return {"q": [b.get_state(i) for i in range(state["count"])], "t": t, "gamma": gamma}
    s = state["solver"]
    if op == "rhs":
        dq, rate = s.rhs(state["q"], want_E=True)
        return {"dq": dq, "rate": rate}
    if op == "relax_step":
        gk, g, out = s.relax_step(state["u"], state["u_new"], state["deta"])
        return {"gamma_elem": gk, "gamma": g, "q": out}
    q = state["q"].clone()  # every pass starts from the stored initial state, as a restart or a sweep does
    if op == "estimate":
        return dict(s.step_estimate(q, state["dt"]), q=q)
    t, hist, gk = s.advance(q, state["case"]["steps"], state["dt"])
    return {"q": q, "t": t, "gamma": hist, "gamma_elem": gk}


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without

def work(case):
    """Bytes: inputs once and outputs once.  Flops: every pair of an LGL line once (two-point
    flux 56, accumulation 20), face fluxes 56 + 55, stage states 40, entropy increments 122, the
    relaxation 140 per node, and per Navier--Stokes stage the D products of gradient and divergence."""
    stages = STAGES[case["rk"]]
    if case["op"] == "batch":
        rng = np.random.default_rng(case["count"] * 1000 + case["nmax"])
        sizes = [(int(rng.integers(4, case["nmax"] + 1)), int(rng.integers(2, 6))) for _ in range(case["count"])]
        meshes = [(n ** 3, p) for n, p in sizes]
    else:
        meshes = [(case["nx"] * case["ny"] * case["nz"], case["p"])]
    if case["op"] == "rhs":
        stages, extra = 1, 40.0
    else:
        extra = 40.0 + 122.0 * (stages - 1) / stages + 140.0 / stages
    flops = bytes_ = 0.0
    for k, p in meshes:
        p1 = p + 1
        nodes = k * p1 ** 3
        if case["op"] == "relax_step":
            flops += 140.0 * nodes
            bytes_ += nodes * 120.0 + k * 16.0
            continue
        line = p1 * p / 2 * 76.0 + 2 * 5 * p1 + (56.0 + 55.0) + 10.0
        if case["mu"] > 0.0:
            line += 2 * 4 * (2.0 * p1 * p1 + 8.0)
            extra_ns = 90.0
        else:
            extra_ns = 0.0
        flops += (3.0 * k * p1 * p1 * line + nodes * (extra + extra_ns)) * stages * case.get("steps", 1)
        bytes_ += nodes * 80.0 + k * (32.0 if case["op"] == "estimate" else 8.0)
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------------------------------------
# the scheme in plain torch FP64

def _l1pmx(z):
    """log(1 + z) - z without cancellation for small z (Taylor below 0.02)."""
    s = torch.zeros_like(z)
    for k in range(13, 1, -1):
        s = s * z + (-1.0) ** (k + 1) / k
    return torch.where(z.abs() < 0.02, s * z * z, torch.log1p(z) - z)


def _entropy_vars(q):
    v = q[1:4] / q[0]
    v2 = (v * v).sum(0)
    pr = (GAMMA - 1.0) * (q[4] - 0.5 * q[0] * v2)
    s = torch.log(pr) - GAMMA * torch.log(q[0])
    beta = q[0] / pr
    return torch.stack([(GAMMA - s) / (GAMMA - 1.0) - 0.5 * beta * v2, beta * v[0], beta * v[1], beta * v[2], -beta])


def _increments(q, e):
    """x = d rho/rho, y = d p/p, the velocity change and rho'/rho of the increment e, without cancellation."""
    rho, v = q[0], q[1:4] / q[0]
    pr = (GAMMA - 1.0) * (q[4] - 0.5 * rho * (v * v).sum(0))
    rho1 = rho + e[0]
    dv = (e[1:4] - v * e[0]) / rho1
    y = (GAMMA - 1.0) * (e[4] - (v * e[1:4]).sum(0) + 0.5 * (v * v).sum(0) * e[0] - 0.5 * rho1 * (dv * dv).sum(0)) / pr
    return e[0] / rho, y, v, dv, rho, pr


def mesh_sum(mesh, a):
    return (a * mesh.mass).sum((-3, -2, -1))


def _breg(q, gd, mesh):
    """Element sums of S(q + gd) - S(q) - w(q).gd and of its derivative along gd."""
    x, y, v, dv, rho, pr = _increments(q, gd)
    opx = 1.0 + x
    lx, ly = _l1pmx(x), _l1pmx(y)
    kin = 0.5 * rho * opx * rho / pr * (dv * dv).sum(0)
    val = rho * ((GAMMA * (opx * lx + x * x) - ly - x * (y + ly)) / (GAMMA - 1.0)) + kin
    der = (_increment_vars(q, gd) * gd).sum(0)
    return mesh_sum(mesh, val), mesh_sum(mesh, der)


def _increment_vars(q, e):
    """w(q + e) - w(q) without cancellation."""
    x, y, v, dv, rho, pr = _increments(q, e)
    beta = rho / pr
    ds = (y + _l1pmx(y)) - GAMMA * (x + _l1pmx(x))
    opx = 1.0 + x
    db = (x - y) / (1.0 + y)
    v2 = (v * v).sum(0)
    dk = (x - y) * v2 + opx * (2.0 * (v * dv).sum(0) + (dv * dv).sum(0))
    return torch.stack([-ds / (GAMMA - 1.0) - 0.5 * beta * dk / (1.0 + y)]
                       + [beta * ((x - y) * v[k] + opx * dv[k]) / (1.0 + y) for k in range(3)] + [-beta * db])


class _Reference:
    def __init__(self, mesh, case):
        self.mesh, self.diss, self.mu = mesh, case["diss"], case["mu"]
        self.flow = case.get("flow")
        self.kappa = self.mu * GAMMA / ((GAMMA - 1.0) * (SHOCK[2] if self.flow == "shock" else 0.72))

    # exterior conserved state on the x faces at time t, or None
    def outside(self, side, t):
        if self.flow == "sod":
            return torch.tensor(_sod_ends()[5 * side:5 * side + 5], device=_device(), dtype=torch.float64)
        if self.flow == "shock":
            x = torch.tensor([self.mesh.hi[0] if side else self.mesh.lo[0]], device=_device(), dtype=torch.float64)
            return _conserved(*_shock_state(x, t))[:, 0]
        return None

    @staticmethod
    def param(q):
        v = q[1:4] / q[0]
        pr = (GAMMA - 1.0) * (q[4] - 0.5 * q[0] * (v * v).sum(0))
        z1 = torch.sqrt(q[0] / pr)
        return torch.stack([z1, z1 * v[0], z1 * v[1], z1 * v[2], torch.sqrt(q[0] * pr)])

    @staticmethod
    def logmean_parts(a, b):
        """(S/2)/lnmean and its inverse."""
        r = (a - b) / (a + b)
        u = r * r
        f = 1.0 + u * (1.0 / 3 + u * (1.0 / 5 + u * (1.0 / 7 + u * (1.0 / 9 + u * (1.0 / 11 + u / 13)))))
        f = torch.where(u < 2.5e-3, f, torch.log(a / b) / (2.0 * torch.where(u < 2.5e-3, torch.ones_like(r), r)))
        return f

    def flux(self, a, b, m):
        s1, s5 = a[0] + b[0], a[4] + b[4]
        f1, f5 = self.logmean_parts(a[0], b[0]), self.logmean_parts(a[4], b[4])
        rho = 0.25 * s1 * s5 / f5
        u = [(a[k] + b[k]) / s1 for k in (1, 2, 3)]
        p1 = s5 / s1
        c1, c2 = (GAMMA + 1.0) / (2.0 * GAMMA), (GAMMA - 1.0) / (2.0 * GAMMA)
        p2 = p1 * (c1 * f1 / f5 + c2)
        mass = rho * u[m]
        f = [mass] + [mass * u[k] for k in range(3)]
        f[1 + m] = f[1 + m] + p1
        f.append(u[m] * GAMMA / (GAMMA - 1.0) * p2 + 0.5 * mass * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]))
        return torch.stack(f)

    @staticmethod
    def conserved(z):
        rho, pr = z[0] * z[4], z[4] / z[0]
        return _conserved(rho, [z[k] / z[0] for k in (1, 2, 3)], pr)

    def face_flux(self, a, b, m):
        f = self.flux(a, b, m)
        if self.diss == 1:
            lam = torch.maximum(*[(z[1 + m].abs() + math.sqrt(GAMMA)) / z[0] for z in (a, b)])
            f = f - 0.5 * lam * (self.conserved(b) - self.conserved(a))
        elif self.diss == 2:
            f = f - 0.5 * self.matrix(a, b, m)
        return f

    def matrix(self, a, b, m):
        """R |Lambda| T R^T [[w]] at the mean parameter vector (Barth-scaled eigenvectors)."""
        zb = 0.5 * (a + b)
        rho, pr = zb[0] * zb[4], zb[4] / zb[0]
        u = [zb[k] / zb[0] for k in (1, 2, 3)]
        c = math.sqrt(GAMMA) / zb[0]
        k2 = 0.5 * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2])
        h = c * c / (GAMMA - 1.0) + k2
        ds = -(GAMMA + 1.0) * torch.log(b[0] / a[0]) - (GAMMA - 1.0) * torch.log(b[4] / a[4])
        jw = [-ds / (GAMMA - 1.0) - 0.5 * sum(b[k] * b[k] - a[k] * a[k] for k in (1, 2, 3))]
        jw += [b[0] * b[k] - a[0] * a[k] for k in (1, 2, 3)] + [a[0] * a[0] - b[0] * b[0]]
        one, zero = torch.ones_like(c), torch.zeros_like(c)
        un = u[m]
        vecs = []
        for sgn in (-1.0, 1.0):
            vecs.append((torch.stack([one] + [u[k] + (sgn * c if k == m else 0.0) for k in range(3)] + [h + sgn * un * c]),
                         (un + sgn * c).abs() * rho / (2.0 * GAMMA)))
        vecs.append((torch.stack([one] + u + [k2]), un.abs() * rho * (GAMMA - 1.0) / GAMMA))
        for t in range(3):
            if t != m:
                vecs.append((torch.stack([zero] + [one if k == t else zero for k in range(3)] + [u[t]]), un.abs() * pr))
        out = 0.0
        for r, scale in vecs:
            out = out + r * (scale * sum(r[k] * jw[k] for k in range(5)))
        return out

    def next_trace(self, left, m, value):
        """Left traces of the +x_m neighbours (a prescribed value beyond the last element)."""
        ax = 3 - m
        out = torch.roll(left, -1, ax)
        if value is not None:
            out.select(ax, out.shape[ax] - 1).copy_(value.reshape(-1, 1, 1, 1, 1).expand_as(out.select(ax, 0)))
        return out

    def prev_trace(self, right, m, value):
        ax = 3 - m
        out = torch.roll(right, 1, ax)
        if value is not None:
            out.select(ax, 0).copy_(value.reshape(-1, 1, 1, 1, 1).expand_as(out.select(ax, 0)))
        return out

    def rhs(self, q, t):
        mesh, p = self.mesh, self.mesh.p
        z = self.param(q)
        out = torch.zeros_like(q)
        for m in range(3):
            zm, om = z.movedim(6 - m, 0), out.movedim(6 - m, 0)
            s = 2.0 / mesh.h[m]
            for i in range(p + 1):
                for j in range(i + 1, p + 1):
                    f = self.flux(zm[i], zm[j], m)
                    om[i] -= s * 2.0 * mesh.D[i, j] * f
                    om[j] -= s * 2.0 * mesh.D[j, i] * f
            qb = [self.outside(k, t) if m == 0 else None for k in (0, 1)]
            zb = [None if v is None else self.param(v) for v in qb]
            fr = self.face_flux(zm[p], self.next_trace(zm[0], m, zb[1]), m)
            fl = torch.roll(fr, 1, 3 - m)
            if zb[0] is not None:
                fl = self.face_flux(self.prev_trace(zm[p], m, zb[0]), zm[0], m)
            # the strong-form diagonal 2 D_pp f(q) = f(q)/omega_p cancels against the SAT's own flux
            om[p] -= s / mesh.w[p] * fr
            om[0] += s / mesh.w[0] * fl
        if self.mu > 0.0:
            self.viscous(q, t, out)
        return out

    def viscous(self, q, t, out):
        mesh, p = self.mesh, self.mesh.p
        w = _entropy_vars(q)
        D = torch.tensor(mesh.D, device=_device())
        theta = []
        for m in range(3):
            wm = w.movedim(6 - m, 0)
            g = torch.einsum("ij,j...->i...", D, wm)
            qb = [self.outside(k, t) if m == 0 else None for k in (0, 1)]
            wb = [None if v is None else _entropy_vars(v) for v in qb]
            g[p] += 0.5 * (self.next_trace(wm[0], m, wb[1]) - wm[p]) / mesh.w[p]
            g[0] -= 0.5 * (self.prev_trace(wm[p], m, wb[0]) - wm[0]) / mesh.w[0]
            theta.append((2.0 / mesh.h[m] * g).movedim(0, 6 - m))
        v = q[1:4] / q[0]
        a = -1.0 / w[4]
        dv = [[a * (theta[m][1 + k] + v[k] * theta[m][4]) for k in range(3)] for m in range(3)]
        div = dv[0][0] + dv[1][1] + dv[2][2]
        for m in range(3):
            tau = [self.mu * (dv[m][k] + dv[k][m] - (2.0 / 3.0 * div if k == m else 0.0)) for k in range(3)]
            F = torch.stack(tau + [tau[0] * v[0] + tau[1] * v[1] + tau[2] * v[2] + self.kappa * a * a * theta[m][4]])
            Fm = F.movedim(6 - m, 0)
            dF = torch.einsum("ij,j...->i...", D, Fm)
            nxt, prv = torch.roll(Fm[0], -1, 3 - m), torch.roll(Fm[p], 1, 3 - m)
            if m == 0 and self.flow in ("sod", "shock"):  # boundary faces take the interior viscous flux
                nxt.select(3, -1).copy_(Fm[p].select(3, -1))
                prv.select(3, 0).copy_(Fm[0].select(3, 0))
            dF[p] += 0.5 * (nxt - Fm[p]) / mesh.w[p]
            dF[0] -= 0.5 * (prv - Fm[0]) / mesh.w[0]
            out[1:] += 2.0 / mesh.h[m] * dF.movedim(0, 6 - m)

    def entropies(self, q):
        pr = (GAMMA - 1.0) * (q[4] - 0.5 * (q[1:4] * q[1:4]).sum(0) / q[0])
        return mesh_sum(self.mesh, -q[0] * (torch.log(pr) - GAMMA * torch.log(q[0])) / (GAMMA - 1.0))

    def roots(self, q, d, A, floor):
        """gamma_kappa > 0 of sum P D(gamma) + gamma A = 0 (Newton from the right; +inf: unconstrained)."""
        mesh = self.mesh
        x, y, _, _, rho, pr = _increments(q, d)
        v = q[1:4] / q[0]
        y0 = (GAMMA - 1.0) * (d[4] - (v * d[1:4]).sum(0) + 0.5 * (v * v).sum(0) * d[0]) / pr
        dv = (d[1:4] - v * d[0]) / rho
        a = mesh_sum(mesh, 0.5 * rho * (x * x + (x - y0) ** 2 / (GAMMA - 1.0) + rho / pr * (dv * dv).sum(0)))
        free = ~(torch.sqrt(2.0 * a / mesh_sum(mesh, rho)) > floor)
        g = torch.where(free, torch.ones_like(a), (-A / a).clamp(1e-3, 8.0))
        for _ in range(25):
            gd = g[..., None, None, None] * d
            val, der = _breg(q, gd, mesh)
            slope = der / g + A
            step = torch.where(slope > 0.0, (val + g * A) / slope, -g)
            g = torch.where(free, g, (g - step).clamp(1e-3, 8.0))
        return torch.where(free, torch.full_like(g, math.inf), g)

    def step(self, q, dt, t, tab, floor):
        a, b, c = tab
        ks, A = [], 0.0
        for i in range(len(b)):
            e = torch.zeros_like(q)
            for j in range(i):
                if a[i][j] != 0.0:
                    e = e + dt * a[i][j] * ks[j]
            ks.append(self.rhs(q + e, t + c[i] * dt))
            if i > 0 and b[i] != 0.0:
                A = A - dt * b[i] * mesh_sum(self.mesh, (_increment_vars(q, e) * ks[i]).sum(0))
        d = sum(dt * b[i] * ks[i] for i in range(len(b)) if b[i] != 0.0)
        gk = self.roots(q, d, A, floor)
        g = float(gk.min())
        return d, A, gk, g if math.isfinite(g) else 1.0


TABLEAUX = {
    "bs3": ([[], [0.5], [0.0, 0.75]], [2.0 / 9, 1.0 / 3, 4.0 / 9], [0.0, 0.5, 0.75]),
    "rk4": ([[], [0.5], [0.0, 0.5], [0.0, 0.0, 1.0]], [1.0 / 6, 1.0 / 3, 1.0 / 3, 1.0 / 6], [0.0, 0.5, 0.5, 1.0]),
    "rk65": ([[], [0.25], [0.125, 0.125], [0.0, -0.5, 1.0], [3.0 / 16, 0.0, 0.0, 9.0 / 16],
              [-3.0 / 7, 2.0 / 7, 12.0 / 7, -12.0 / 7, 8.0 / 7]],
             [7.0 / 90, 0.0, 32.0 / 90, 12.0 / 90, 32.0 / 90, 7.0 / 90], [0.0, 0.25, 0.25, 0.5, 0.75, 1.0]),
}


def _march(ref, q, dt, case):
    floor = 4e-6 if case["precision"] in ("mixed", "mixed_ff") else 1e-8
    t, hist, gk = 0.0, [], None
    for _ in range(case["steps"]):
        d, _, gk, g = ref.step(q, dt, t, TABLEAUX[case["rk"]], floor)
        q, t = q + g * d, t + g * dt
        hist.append(g)
    return q, t, hist, gk


def exact(case, seed):
    if case["op"] == "batch":
        qs, ts, gs = [], [], []
        for mesh, q, dt in _instances(case, seed):
            q, t, hist, _ = _march(_Reference(mesh, case), q, dt, case)
            qs.append(q.reshape(5, mesh.K, mesh.Np))
            ts.append(t)
            gs.append(hist[-1])
        return {"q": qs, "t": np.array(ts), "gamma": np.array(gs)}
    if case["op"] == "relax_step":
        mesh, u, u_new, deta = _relax_inputs(case, seed)
        d = u_new - u
        A = mesh_sum(mesh, (_entropy_vars(u) * d).sum(0)) - deta
        gk = _Reference(mesh, case).roots(u, d, A, 1e-8)
        g = gk.min()
        return {"gamma_elem": gk.reshape(-1), "gamma": g.reshape(1), "q": (u + g * d).reshape(5, mesh.K, mesh.Np)}
    mesh = _Mesh(case["flow"], case["p"], (case["nx"], case["ny"], case["nz"]))
    ref = _Reference(mesh, case)
    q = _state(case["flow"], mesh, seed)
    shape = (5, mesh.K, mesh.Np)
    if case["op"] == "rhs":
        dq = ref.rhs(q, 0.0)
        return {"dq": dq.reshape(shape), "rate": mesh_sum(mesh, (_entropy_vars(q) * dq).sum(0)).reshape(-1)}
    dt = _dt(q, mesh, case["mu"])
    if case["op"] == "estimate":
        d, A, gk, g = ref.step(q, dt, 0.0, TABLEAUX[case["rk"]], 4e-6 if "mixed" in case["precision"] else 1e-8)
        new = q + g * d
        scalar = lambda v: torch.tensor([v], dtype=torch.float64, device=_device())  # noqa: E731
        return {"eta_old": ref.entropies(q).reshape(-1),
                "deta": (mesh_sum(mesh, (_entropy_vars(q) * d).sum(0)) - A).reshape(-1),
                "eta_new": ref.entropies(new).reshape(-1), "gamma_elem": gk.reshape(-1),
                "gamma": scalar(g), "t": scalar(g * dt), "q": new.reshape(shape)}
    q, t, hist, gk = _march(ref, q, dt, case)
    one = lambda v: torch.tensor(v, dtype=torch.float64, device=_device())  # noqa: E731
    return {"q": q.reshape(shape), "t": one([t]), "gamma": one(hist), "gamma_elem": gk.reshape(-1)}
