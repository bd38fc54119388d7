"""What a user of the framework has it do: residuals, Runge-Kutta steps, vector-Jacobian products and
trajectory gradients through the public Solver, over the degrees, mesh sizes, precisions and options
that the repository's tests, benchmark and studies use.

The meshes and states here are made from the seed in plain torch, and exact() evaluates the same
discretisation in plain float64 torch, so neither depends on the code being measured.
"""
from __future__ import annotations

import math

import numpy as np
import torch

GAMMA, PR = 1.4, 0.72
# flow: box, Mach number, Reynolds number of the viscous form
FLOWS = {
    "tgv": ((-math.pi, math.pi), 0.1, 1600.0),        # Taylor-Green vortex with developed perturbations
    "vortex": ((-5.0, 5.0), 0.5, 1000.0),             # isentropic vortex
    "mms": ((0.0, 1.0), 800.0 / math.sqrt(1.4e5), 4.0e6),   # bounded supersonic box with Dirichlet data and a source
}


def _case(name, op, p, k, flow="tgv", prec="fp64", warp=0.0, visc=True, flux="esc", diss=True, steps=1):
    c = {"op": op, "p": p, "kx": k[0], "ky": k[1], "kz": k[2], "flow": flow, "prec": prec, "warp": warp,
         "visc": visc, "flux": flux, "diss": diss, "steps": steps}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one residual of the 4^3 Taylor-Green box, bound by launches and latency
        _case("rhs_p3_4cubed", "rhs", 3, (4, 4, 4)),
        # the 4^3 box advanced ten steps in one call, inviscid, with its budgets (entropy check runs)
        _case("steps_p3_4cubed_inviscid", "step", 3, (4, 4, 4), visc=False, steps=10),
        # the ordinary float64 residual on a curved mesh
        _case("rhs_p4_16cubed_warped", "rhs", 4, (16, 16, 16), warp=0.1),
        # a low degree on a ragged box with many small elements
        _case("rhs_p2_41x37x39", "rhs", 2, (41, 37, 39)),
        # the split-form flux on a ragged bounded box with Dirichlet data and a source, two steps at a time
        _case("steps_p3_mms_kg", "step", 3, (15, 17, 13), flow="mms", warp=0.05, flux="kg", steps=2),
        # the differentiation workload: vector-Jacobian product and trajectory gradient of the vortex
        _case("vjp_p4_8cubed_vortex", "vjp", 4, (8, 8, 8), flow="vortex", warp=0.1),
        _case("grad_p4_8cubed_vortex", "grad", 4, (8, 8, 8), flow="vortex", warp=0.1, steps=3),
        # the highest degree of the per-element kernels: steps with budgets in both precisions
        _case("step_p7_24cubed", "step", 7, (24, 24, 24)),
        _case("step_fp32_p7_24cubed", "step", 7, (24, 24, 24), prec="fp32"),
        # float32-mixed: many small steps on the curved mesh, and one residual at a middle degree
        _case("steps_fp32_p4_16cubed", "step", 4, (16, 16, 16), prec="fp32", warp=0.1, steps=5),
        _case("rhs_fp32_p5_21x23x22", "rhs", 5, (21, 23, 22), flow="vortex", prec="fp32"),
        # the highest degree of the cost comparison
        _case("rhs_p15_6x5x7", "rhs", 15, (6, 5, 7)),
    ]


def draw(rng):
    """One more case: any operation, degree and option combination above on a box of random, often
    odd element counts; sizes spread over the logarithm of the work."""
    op = rng.choice(["rhs", "rhs", "step", "step", "vjp", "grad"])
    p = rng.choice([1, 2, 3, 3, 4, 4, 5, 6, 7, 7] + ([15] if op == "rhs" else []))
    prec = "fp32" if op in ("rhs", "step") and p < 15 and rng.random() < 0.35 else "fp64"
    flow = rng.choice(["tgv", "tgv", "vortex"] + (["mms"] if p < 8 else []))
    flux = "esc" if rng.random() < 0.7 else ("kg" if prec == "fp32" else rng.choice(["kg", "dc"]))
    steps = {"rhs": 1, "vjp": 1, "step": rng.choice([1, 2, 5, 10]), "grad": rng.choice([1, 2, 3])}[op]
    evals = {"rhs": 1, "vjp": 3, "step": 6 * steps, "grad": 26 * steps}[op] / (10.0 if prec == "fp32" else 1.0)
    N3 = (p + 1) ** 3
    most = min(7.0e6, 2.0e7 / evals) if op != "grad" else 6.0e4
    nodes = math.exp(rng.uniform(math.log(3.0e3), math.log(most)))
    side = max(2.0, (nodes / N3) ** (1.0 / 3.0))
    k = tuple(max(2, round(side * rng.uniform(0.8, 1.2))) for _ in range(3))
    return _case(None, op, p, k, flow, prec, rng.choice([0.0, 0.05, 0.1]), rng.random() < 0.75, flux,
                 flux != "esc" or rng.random() < 0.8, steps)


# -- inputs

def _lgl(p):
    """Legendre-Gauss-Lobatto nodes and weights: the roots of (1 - x^2) P_p'(x)."""
    P = np.polynomial.legendre.Legendre.basis(p)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    for _ in range(4):
        x[1:-1] -= P.deriv()(x[1:-1]) / P.deriv(2)(x[1:-1])
    x = 0.5 * (x - x[::-1])
    return x, 2.0 / (p * (p + 1) * P(x) ** 2)


def _coords(case, seed):
    """Node coordinates [K, 3, N, N, N] of the box, warped sinusoidally with phases from the seed."""
    (lo, hi), N = FLOWS[case["flow"]][0], case["p"] + 1
    k = (case["kx"], case["ky"], case["kz"])
    xi = torch.tensor(_lgl(case["p"])[0], device="cuda")
    e = torch.arange(k[0] * k[1] * k[2], device="cuda")
    idx = (e % k[0], (e // k[0]) % k[1], e // (k[0] * k[1]))
    h = [(hi - lo) / n for n in k]
    x = torch.empty((e.numel(), 3, N, N, N), dtype=torch.float64, device="cuda")
    for d in range(3):
        shape = [-1, 1, 1, 1]
        shape[3 - d] = N
        x[:, d] = (lo + (idx[d][:, None] + 0.5 * (xi[None] + 1.0)) * h[d]).reshape(shape)
    if case["warp"]:
        phi = np.random.default_rng(seed).uniform(0.0, 2.0 * math.pi, (3, 3))
        s = [[torch.sin(2.0 * math.pi * (x[:, m] - lo) / (hi - lo) + phi[i, m]) for m in range(3)] for i in range(3)]
        for i in range(3):
            x[:, i] += case["warp"] * h[i] * s[i][0] * s[i][1] * s[i][2]
    return x


def _state(case, x, seed):
    """Conserved state [K, 5, N, N, N]: the flow at a random phase with a few smooth random modes in
    density, velocity and temperature, as a flow that has developed for a while has."""
    (lo, hi), Ma, _ = FLOWS[case["flow"]]
    R = 1.0 / (GAMMA * Ma * Ma)
    rng = np.random.default_rng(seed + 1000003)
    X = [2.0 * math.pi * (x[:, d] - lo) / (hi - lo) for d in range(3)]

    def modes(amp, n=3):
        f = 0.0
        for _ in range(n):
            w = rng.integers(-2, 3, 3)
            f = f + amp * rng.normal() * torch.sin(w[0] * X[0] + w[1] * X[1] + w[2] * X[2] + rng.uniform(0, 2 * math.pi))
        return f

    if case["flow"] == "tgv":
        a = [X[d] + rng.uniform(0, 2 * math.pi) for d in range(3)]
        u = [torch.sin(a[0]) * torch.cos(a[1]) * torch.cos(a[2]) + modes(0.05),
             -torch.cos(a[0]) * torch.sin(a[1]) * torch.cos(a[2]) + modes(0.05), modes(0.05)]
        rho = 1.0 + GAMMA * Ma * Ma / 16.0 * (torch.cos(2 * a[0]) + torch.cos(2 * a[1])) * (torch.cos(2 * a[2]) + 2.0) + modes(0.01)
        T = 1.0 + modes(0.01)
    elif case["flow"] == "vortex":
        beta, n = 5.0, 1.0 / math.sqrt(3.0)
        d = [x[:, m] - rng.uniform(-1, 1) for m in range(3)]
        ax = n * (d[0] + d[1] + d[2])
        r = [d[m] - n * ax for m in range(3)]
        s = beta / (2 * math.pi) * torch.exp(0.5 * (1.0 - r[0] ** 2 - r[1] ** 2 - r[2] ** 2))
        u = [n * s * (r[(m + 2) % 3] - r[(m + 1) % 3]) + (1 / math.sqrt(2), -1 / math.sqrt(2), 0.0)[m] + modes(0.01) for m in range(3)]
        T = 1.0 - 0.5 * (GAMMA - 1.0) * Ma * Ma * s * s + modes(0.005)
        rho = T ** (1.0 / (GAMMA - 1.0)) * (1.0 + modes(0.005))
    else:
        rho = 1.0 + modes(0.05)
        u = [1.0 + modes(0.03) for _ in range(3)]
        T = 1.0 + modes(0.05)
    q = torch.empty((x.shape[0], 5) + tuple(x.shape[2:]), dtype=torch.float64, device=x.device)
    q[:, 0] = rho
    for m in range(3):
        q[:, 1 + m] = rho * u[m]
    q[:, 4] = rho * R * T / (GAMMA - 1.0) + 0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
    return q


def _dt(case):
    """A fixed step at an acoustic CFL number of about 0.5."""
    (lo, hi), Ma, _ = FLOWS[case["flow"]]
    return 0.5 * (hi - lo) / max(case["kx"], case["ky"], case["kz"]) / ((case["p"] + 1) ** 2 * (1.0 / Ma + 2.0))


def _reynolds(case):
    return FLOWS[case["flow"]][2] if case["visc"] else 0.0


def _inputs(case, seed):
    x = _coords(case, seed)
    q = _state(case, x, seed)
    ext = src = lam = None
    if case["flow"] == "mms":
        ext = q.clone()
        g = torch.Generator(device="cuda").manual_seed(seed)
        src = torch.randn(q.shape[:2] + (1, 1, 1), generator=g, dtype=torch.float64, device="cuda") * torch.ones_like(q)
    if case["op"] == "vjp":
        # the cotangent a kinetic-energy functional hands back: P J (-|u|^2/2, u, 0) on the unwarped elements
        (lo, hi), w = FLOWS[case["flow"]][0], torch.tensor(_lgl(case["p"])[1], device="cuda")
        vol = (hi - lo) ** 3 / (8.0 * case["kx"] * case["ky"] * case["kz"])
        u = q[:, 1:4] / q[:, :1]
        lam = torch.zeros_like(q)
        lam[:, 0] = -0.5 * (u * u).sum(1)
        lam[:, 1:4] = u
        lam *= vol * w.view(-1, 1, 1) * w.view(1, -1, 1) * w
    return x, q, ext, src, lam


def prepare(case, seed):
    from paper_1911_10966_gb300 import Solver
    x, q, ext, src, lam = _inputs(case, seed)
    (lo, hi), Ma, _ = FLOWS[case["flow"]]
    s = Solver(case["p"], case["kx"], case["ky"], case["kz"], x.cpu().numpy(), Ma=Ma, Re=_reynolds(case), lo=(lo,) * 3,
               hi=(hi,) * 3, dissipation=case["diss"], precision=case["prec"], volume_flux=case["flux"],
               bounded=(case["flow"] == "mms",) * 3)
    if ext is not None:
        s.set_exterior(ext)
        s.set_source(src)
    st = {"case": case, "solver": s, "q": q, "dt": _dt(case), "lam": lam}
    if case["op"] == "step":
        st["work"] = torch.empty_like(q)
        st["budgets"] = torch.zeros(5, dtype=torch.float64, device="cuda")
    if case["op"] == "grad":
        st["mu"] = torch.tensor(s.mu, dtype=torch.float64)
    return st


def run(st):
    case, s, q = st["case"], st["solver"], st["q"]
    if case["op"] == "rhs":
        return s.rhs(q)
    if case["op"] == "step":
        w = st["work"].copy_(q)
        s.rk_step(w, st["dt"], case["steps"])
        s.budgets_async(w, st["budgets"])
        return {"q": w, "budgets": st["budgets"]}
    if case["op"] == "vjp":
        if case["visc"]:
            g, gmu = s.rhs_vjp(q, st["lam"], want_mu=True)
            return {"grad": g, "grad_mu": gmu}
        return {"grad": s.rhs_vjp(q, st["lam"])}
    from paper_1911_10966_gb300.autograd import KineticEnergy, Trajectory
    q0 = q.clone().requires_grad_(True)
    mu = st["mu"].clone().requires_grad_(True)
    ke = KineticEnergy.apply(Trajectory.apply(q0, mu, s, st["dt"], case["steps"]), s)
    ke.backward()
    out = {"ke": ke.detach(), "grad": q0.grad}
    if case["visc"]:
        out["grad_mu"] = mu.grad
    return out


def work(case):
    """Floating-point operations of the discretisation (one per +, -, *, division, logarithm; two per
    multiply-add) and the bytes of state, geometry and result, each once per residual."""
    N, nodes = case["p"] + 1, case["kx"] * case["ky"] * case["kz"] * (case["p"] + 1) ** 3
    f = {"esc": 82.0 * 1.5 * case["p"], "kg": 56.0 * 1.5 * case["p"], "dc": 75.0 + 30.0 * N}[case["flux"]]
    f += 57.0 + 140.0 * 6.0 / N + (223.0 + 48.0 * N + 96.0 / N if case["visc"] else 0.0)
    w = 4 if case["prec"] == "fp32" else 8
    b = 5 * 8 + 10 * w + 5 * w
    evals = {"rhs": 1, "step": 6 * case["steps"], "vjp": 2, "grad": (6 + 12) * case["steps"]}[case["op"]]
    return {"bytes": float(b * evals * nodes), "flops": float(f * evals * nodes)}


# -- the same discretisation in plain float64 torch

def _log_mean(a, b):
    """(a - b)/log(a/b), by the artanh series for close arguments."""
    s = a + b
    f = (a - b) / s
    u = f * f
    near = u < 1e-3
    un, fs = torch.where(near, u, torch.zeros_like(u)), torch.where(near, torch.full_like(f, 0.5), f)
    ser = 1.0 + un * (1 / 3 + un * (1 / 5 + un * (1 / 7 + un * (1 / 9 + un * (1 / 11 + un / 13)))))
    return 0.5 * s / torch.where(near, ser, torch.atanh(fs) / fs)


class _Plain:
    def __init__(self, case, x, ext, src, mu=None):
        self.c, self.N, self.src = case, case["p"] + 1, src
        (_, _), Ma, _ = FLOWS[case["flow"]]
        xi, w = _lgl(case["p"])
        N = self.N
        bw = np.array([1.0 / np.prod([xi[i] - xi[j] for j in range(N) if j != i]) for i in range(N)])
        D = np.array([[0.0 if i == j else bw[j] / bw[i] / (xi[i] - xi[j]) for j in range(N)] for i in range(N)])
        D -= np.diag(D.sum(1))
        self.D, self.w = torch.tensor(D, device="cuda"), torch.tensor(w, device="cuda")
        self.R = 1.0 / (GAMMA * Ma * Ma)
        self.mu = mu if mu is not None else (1.0 / _reynolds(case) if case["visc"] else 0.0)
        k = (case["kx"], case["ky"], case["kz"])
        e = torch.arange(k[0] * k[1] * k[2], device="cuda")
        c = [e % k[0], (e // k[0]) % k[1], e // (k[0] * k[1])]
        self.nbr, self.wall = [], []
        for l in range(3):
            for d in (-1, 1):
                m = list(c)
                m[l] = (c[l] + d) % k[l]
                self.nbr.append(m[0] + k[0] * (m[1] + k[1] * m[2]))
                out = (c[l] + d < 0) | (c[l] + d >= k[l])
                self.wall.append((out & (case["flow"] == "mms")).view(-1, 1, 1, 1))
        self.ext = ext
        x = x - x[:, :, :1, :1, :1]
        dX = [[self.dl(x[:, m], a) for a in range(3)] for m in range(3)]
        self.J = (dX[0][0] * (dX[1][1] * dX[2][2] - dX[1][2] * dX[2][1]) - dX[0][1] * (dX[1][0] * dX[2][2] - dX[1][2] * dX[2][0])
                  + dX[0][2] * (dX[1][0] * dX[2][1] - dX[1][1] * dX[2][0]))
        self.Ja = [[None] * 3 for _ in range(3)]
        for m in range(3):
            v = [x[:, (m + 2) % 3] * dX[(m + 1) % 3][j] for j in range(3)]
            for l in range(3):
                a, b = (l + 1) % 3, (l + 2) % 3
                self.Ja[l][m] = self.dl(v[a], b) - self.dl(v[b], a)

    def dl(self, u, l):
        return torch.einsum("ij,...j->...i", self.D, u.movedim(-1 - l, -1)).movedim(-1, -1 - l)

    def face(self, u, l, side):
        return u.select(-1 - l, -1 if side else 0)

    def put(self, out, val, l, side):
        at = torch.zeros(self.N, dtype=torch.float64, device="cuda")
        at[-1 if side else 0] = 1.0
        shape = [1] * out.dim()
        shape[-1 - l] = self.N
        return out + at.view(shape) * val.unsqueeze(out.dim() - 1 - l)

    def prim(self, q):
        rho = q[:, 0]
        u = [q[:, 1 + m] / rho for m in range(3)]
        p = (GAMMA - 1.0) * (q[:, 4] - 0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2))
        return rho, u, p

    def euler(self, P, n):
        rho, u, p = P
        un = u[0] * n[0] + u[1] * n[1] + u[2] * n[2]
        H = GAMMA / (GAMMA - 1.0) * p / rho + 0.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        return [rho * un] + [rho * un * u[m] + p * n[m] for m in range(3)] + [rho * un * H]

    def flux(self, A, B, n):
        (ra, ua, pa), (rb, ub, pb) = A, B
        if self.c["flux"] == "dc":
            return [0.5 * (a + b) for a, b in zip(self.euler(A, n), self.euler(B, n))]
        u = [0.5 * (ua[m] + ub[m]) for m in range(3)]
        un = u[0] * n[0] + u[1] * n[1] + u[2] * n[2]
        qa, qb = ua[0] ** 2 + ua[1] ** 2 + ua[2] ** 2, ub[0] ** 2 + ub[1] ** 2 + ub[2] ** 2
        if self.c["flux"] == "kg":
            f1, pt = 0.5 * (ra + rb) * un, 0.5 * (pa + pb)
            eb = 0.5 * ((pa / ra + pb / rb) / (GAMMA - 1.0) + 0.5 * (qa + qb))
            return [f1] + [f1 * u[m] + pt * n[m] for m in range(3)] + [f1 * eb + pt * un]
        ba, bb = 0.5 * ra / pa, 0.5 * rb / pb
        f1, pt = _log_mean(ra, rb) * un, 0.5 * (ra + rb) / (ba + bb)
        f = [f1] + [f1 * u[m] + pt * n[m] for m in range(3)]
        return f + [f1 * (0.5 / (GAMMA - 1.0) / _log_mean(ba, bb) - 0.25 * (qa + qb)) + u[0] * f[1] + u[1] * f[2] + u[2] * f[3]]

    def volume(self, q, P):
        out = 0.0
        for l in range(3):
            n = self.Ja[l]
            if self.c["flux"] == "dc":
                out = out - self.dl(torch.stack(self.euler(P, n), 1), l)
                continue
            mv = lambda t: t.movedim(-1 - l, -1)  # noqa: E731
            A = [mv(P[0]).unsqueeze(-1), [mv(u).unsqueeze(-1) for u in P[1]], mv(P[2]).unsqueeze(-1)]
            B = [mv(P[0]).unsqueeze(-2), [mv(u).unsqueeze(-2) for u in P[1]], mv(P[2]).unsqueeze(-2)]
            nb = [0.5 * (mv(t).unsqueeze(-1) + mv(t).unsqueeze(-2)) for t in n]
            f = self.flux(A, B, nb)
            out = out - 2.0 * torch.stack([torch.einsum("ij,...ij->...i", self.D, v).movedim(-1, -1 - l) for v in f], 1)
        return out

    def beyond(self, fq, fext, l, side):
        """The far side of face (l, side) of every element: the neighbour's, or the exterior state's at a wall."""
        i = 2 * l + side
        v = self.face(fq, l, 1 - side)[self.nbr[i]]
        return v if fext is None else torch.where(self.wall[i], self.face(fext, l, side), v)

    def rhs(self, q):
        P = self.prim(q)
        out = self.volume(q, P)
        wend = float(self.w[0])
        for l in range(3):
            for side in (0, 1):
                qo, qn = self.face(q, l, side), self.beyond(q, self.ext, l, side)
                A, B = self.prim(qo), self.prim(qn)
                n = [self.face(t, l, side) for t in self.Ja[l]]
                sg = 1.0 if side else -1.0
                val = -sg * (torch.stack(self.flux(A, B, n), 1) - torch.stack(self.euler(A, n), 1))
                if self.c["diss"]:
                    nn = torch.sqrt(n[0] ** 2 + n[1] ** 2 + n[2] ** 2)
                    lam = [(Q[1][0] * n[0] + Q[1][1] * n[1] + Q[1][2] * n[2]).abs() + torch.sqrt(GAMMA * Q[2] / Q[0]) * nn for Q in (A, B)]
                    val = val - 0.5 * torch.maximum(lam[0], lam[1]).unsqueeze(1) * (qo - qn)
                out = self.put(out, val / wend, l, side)
        if self.c["visc"]:
            out = torch.cat([out[:, :1], out[:, 1:] + self.viscous(q, P, wend)], 1)
        out = out / self.J.unsqueeze(1)
        return out if self.src is None else out + self.src

    def viscous(self, q, P, wend):
        rho, u, p = P
        entropy = lambda S: torch.stack([S[0] * S[1][0] / S[2], S[0] * S[1][1] / S[2], S[0] * S[1][2] / S[2], -S[0] / S[2]], 1)  # noqa: E731
        w = entropy(P)
        wx = None if self.ext is None else entropy(self.prim(self.ext))
        th = []
        for l in range(3):
            t = self.dl(w, l)
            for side in (0, 1):
                jump = self.beyond(w, wx, l, side) - self.face(w, l, side)
                t = self.put(t, (0.5 if side else -0.5) * jump / wend, l, side)
            th.append(t)
        g = [sum(self.Ja[a][m].unsqueeze(1) * th[a] for a in range(3)) / self.J.unsqueeze(1) for m in range(3)]
        RT = p / rho
        du = [[RT * (g[m][:, k] + u[k] * g[m][:, 3]) for m in range(3)] for k in range(3)]
        div = du[0][0] + du[1][1] + du[2][2]
        kap = self.mu * GAMMA * self.R / (GAMMA - 1.0) / PR
        F = []
        for m in range(3):
            tau = [self.mu * (du[i][m] + du[m][i] - (2.0 / 3.0 * div if i == m else 0.0)) for i in range(3)]
            F.append(torch.stack(tau + [tau[0] * u[0] + tau[1] * u[1] + tau[2] * u[2] + kap / self.R * RT * RT * g[m][:, 3]], 1))
        out = 0.0
        for l in range(3):
            Ft = sum(self.Ja[l][m].unsqueeze(1) * F[m] for m in range(3))
            out = out + self.dl(Ft, l)
            for side in (0, 1):
                fo = self.face(Ft, l, side)
                fn = torch.where(self.wall[2 * l + side], fo, self.face(Ft, l, 1 - side)[self.nbr[2 * l + side]])
                out = self.put(out, (0.5 if side else -0.5) * (fn - fo) / wend, l, side)
        return out

    def steps(self, q, dt, n):
        """Fixed Dormand-Prince 5 steps."""
        A = [[], [1 / 5], [3 / 40, 9 / 40], [44 / 45, -56 / 15, 32 / 9], [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729],
             [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656]]
        B = [35 / 384, 0.0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84]
        for _ in range(n):
            k = []
            for row in A:
                y = q
                for a, kj in zip(row, k):
                    y = y + dt * a * kj
                k.append(self.rhs(y))
            for b, kj in zip(B, k):
                if b:
                    q = q + dt * b * kj
        return q

    def sums(self, q):
        rho, u, p = self.prim(q)
        PJ = self.w.view(-1, 1, 1) * self.w.view(1, -1, 1) * self.w * self.J
        S = -rho * (torch.log(p) - GAMMA * torch.log(rho)) / (GAMMA - 1.0)
        return (PJ * S).sum(), (PJ * 0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)).sum()


def exact(case, seed):
    x, q, ext, src, lam = _inputs(case, seed)
    if case["op"] in ("rhs", "step"):
        with torch.no_grad():
            m = _Plain(case, x, ext, src)
            if case["op"] == "rhs":
                return m.rhs(q)
            q = m.steps(q, _dt(case), case["steps"])
            S, ke = m.sums(q)
            zero = torch.zeros_like(S)
            return {"q": q, "budgets": torch.stack([S, ke, zero, zero, zero])}
    mu = torch.tensor(1.0 / _reynolds(case) if case["visc"] else 0.0, dtype=torch.float64, device="cuda", requires_grad=True)
    m = _Plain(case, x, ext, src, mu)
    q = q.requires_grad_(True)
    if case["op"] == "vjp":
        y = (m.rhs(q) * lam).sum()
        out = {}
    else:
        y = m.sums(m.steps(q, _dt(case), case["steps"]))[1]
        out = {"ke": y.detach()}
    y.backward()
    out["grad"] = q.grad
    if case["visc"]:
        out["grad_mu"] = mu.grad
    return out
