"""Stretched elements (boxes with one side much longer or shorter than the others), with the flow along the long or
short side only and in every direction: the residual and the vector-Jacobian product lose no more bits than plain
float64 does, whatever the ratio of an element's metric terms.  Bounds: the float64 rounding bound of the other
residual parity tests, with the viscous terms' magnitudes added where there are any; for the gradient with a random
cotangent, whose terms do not cancel, 64 N eps of its largest value for the momentum variables (3 N pair terms of
about ten roundings, on either side), a hundred times that for density and energy, which take differences of
pressure terms c^2/|u|^2 = 100 times the result (up to p = 5: beyond, the two sides' independent metrics differ by
more than that)."""
import math

import numpy as np
import pytest
import torch

from oracle import esdc_oracle as O
from tests.gpu_common import EPS64, assert_parity, geometry_rounding, make_pair, normwise_errors, term_scale

pytestmark = pytest.mark.gpu


def _pair(p, side, flow, flux="esc", Re=0.0, k=(2, 2, 2), Ma=0.1):
    size = [1.0, 1.0, float(side)]
    solver, q, mesh, gas, qo = make_pair(p, k, Ma=Ma, seed=2, Re=Re, box=([0.0] * 3, size), volume_flux=flux)
    x = torch.as_tensor(np.asarray(solver.coords)).reshape(qo.shape[0], 3, *qo.shape[2:])
    X = [2.0 * math.pi * x[:, d] / size[d] for d in range(3)]
    rho = 1.0 + 0.05 * torch.sin(X[0] + 0.3) + 0.05 * torch.cos(X[2]) + 0.03 * torch.sin(X[1])
    T = 1.0 + 0.04 * torch.sin(X[0] + X[2]) + 0.02 * torch.cos(X[1] + 0.5)
    u = [1.0 + 0.3 * torch.sin(X[0] + 0.1) * torch.cos(X[2]) + 0.1 * torch.sin(X[1]),
         0.8 + 0.3 * torch.cos(X[1]) * torch.sin(X[2] + 0.7),
         0.9 + 0.25 * torch.sin(X[0]) * torch.cos(X[1] + 0.2) + 0.1 * torch.cos(X[2])]
    u = [f * u[d] for d, f in enumerate({"x": (1, 0, 0), "z": (0, 0, 1), "all": (1, 1, 1)}[flow])]
    qo = torch.stack([rho] + [rho * v for v in u] + [rho * gas.R * T / (gas.gamma - 1.0) + 0.5 * rho * sum(v * v for v in u)], 1)
    return solver, solver.to_device(qo.numpy()), mesh, gas, qo


@pytest.mark.parametrize("flow", ["x", "z", "all"])
@pytest.mark.parametrize("side", [100.0, 1e3, 1e5, 1e-2, 1e-3, 1e-5])
@pytest.mark.parametrize("p,flux", [(1, "esc"), (3, "esc"), (4, "esc"), (7, "esc"), (3, "kg"), (7, "kg"), (4, "dc"), (7, "dc")])
def test_residual_parity(p, flux, side, flow):
    solver, q, mesh, gas, qo = _pair(p, side, flow, flux)
    assert_parity(solver.rhs(q), O.rhs(qo, mesh, gas, scheme=flux), qo, mesh, gas)


def _viscous_scale(q, mesh, gas):
    """max over nodes of the viscous terms' magnitudes: the viscous residual with every operator entry, metric term
    and factor replaced by its absolute value and every difference by a sum."""
    D, J, A = mesh.sbp.D.abs().clone(), mesh.J, mesh.Ja.abs()          # Ja [K, l, m, ...]
    D[0, 0] += float(1.0 / mesh.sbp.w[0])
    D[-1, -1] += float(1.0 / mesh.sbp.w[0])                            # the lift of a jump of two like values
    dl = lambda f, l: torch.einsum("ij,...j->...i", D, f.movedim(-1 - l, -1)).movedim(-1, -1 - l)  # noqa: E731
    rho, u = q[:, 0], [(q[:, 1 + m] / q[:, 0]).abs() for m in range(3)]
    RT = (gas.gamma - 1.0) * (q[:, 4] - 0.5 * (q[:, 1:4] ** 2).sum(1) / rho) / rho
    w = [v / RT for v in u] + [1.0 / RT]
    th = [[dl(f, a) for f in w] for a in range(3)]
    g = [[sum(A[:, a, m] * th[a][k] for a in range(3)) / J for k in range(4)] for m in range(3)]
    du = [[RT * (g[m][k] + u[k] * g[m][3]) for m in range(3)] for k in range(3)]
    tau = [[gas.mu * (du[i][m] + du[m][i] + (du[0][0] + du[1][1] + du[2][2] if i == m else 0.0)) for m in range(3)] for i in range(3)]
    kap = gas.mu * gas.gamma / (gas.gamma - 1.0) / gas.Pr
    F = [tau[m] + [sum(tau[m][i] * u[i] for i in range(3)) + kap * RT * RT * g[m][3]] for m in range(3)]
    out = [sum(dl(sum(A[:, l, m] * F[m][k] for m in range(3)), l) for l in range(3)) / J for k in range(4)]
    return [0.0] + [float(f.max()) for f in out]


@pytest.mark.parametrize("flow", ["x", "z", "all"])
@pytest.mark.parametrize("side", [100.0, 1e3, 1e-2, 1e-3])
@pytest.mark.parametrize("p,flux", [(2, "esc"), (4, "esc"), (7, "esc"), (3, "kg"), (5, "dc")])
def test_viscous_residual_parity(p, flux, side, flow):
    solver, q, mesh, gas, qo = _pair(p, side, flow, flux, Re=200.0)
    r, ro = solver.rhs(q).cpu(), O.rhs(qo, mesh, gas, scheme=flux)
    T, V = term_scale(qo, mesh, gas), _viscous_scale(qo, mesh, gas)
    for v in range(5):
        err, R = float((r[:, v] - ro[:, v]).abs().max()), float(ro[:, v].abs().max())
        assert err <= max(1e-12 * R, 8.0 * EPS64 * (T[v] + V[v])), (v, err, R, EPS64 * T[v], EPS64 * V[v])


@pytest.mark.parametrize("flow", ["z", "all"])
@pytest.mark.parametrize("side", [30.0, 1e-5])
@pytest.mark.parametrize("flux", ["esc", "kg"])
def test_p15_residual_parity(flux, side, flow):
    """p = 15, with the bound of its other parity tests."""
    solver, q, mesh, gas, qo = _pair(15, side, flow, flux, k=(1, 1, 1))
    assert_parity(solver.rhs(q), O.rhs(qo, mesh, gas, scheme=flux), qo, mesh, gas, geo_rel=geometry_rounding(15))


@pytest.mark.parametrize("k", [(2, 2, 2), (3, 1, 3)])
@pytest.mark.parametrize("side", [4.0, 16.0, 1e3, 1e5, 1e-3, 1e-5])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
def test_vjp_matches_oracle_autograd(p, side, k):
    solver, q, mesh, gas, qo = _pair(p, side, "z", Re=500.0, k=k)
    lam = torch.randn(qo.shape, generator=torch.Generator().manual_seed(11), dtype=torch.float64)
    qq = qo.clone().requires_grad_(True)
    (go,) = torch.autograd.grad(O.rhs(qq, mesh, gas), qq, lam)
    e = normwise_errors(solver.rhs_vjp(q, lam.cuda()), go)
    print("vjp", ["%.1e" % x for x in e])
    assert max(e[1:4]) <= 64 * (p + 1) * EPS64, e
    assert max(e) <= 6400 * (p + 1) * EPS64, e


def test_some_elements_stretched():
    """One thin layer of elements in a box of cubes: its elements take the float64 form, beside the others and in
    the same CTAs, and both forms see each other's faces."""
    for p in (1, 2, 3, 5):
        solver, q, mesh, gas, qo = make_pair(p, (3, 3, 4), seed=3, Re=400.0, noise=1e-2)
        x = np.asarray(solver.coords).reshape(qo.shape[0], 3, *qo.shape[2:]).copy()
        lo, h = -math.pi, 2.0 * math.pi / 4
        z = x[:, 2]                                    # second layer of z thinned to a fiftieth
        f = np.clip((z - (lo + h)) / h, 0.0, 1.0)
        x[:, 2] = z - 0.98 * h * f
        from paper_1911_10966_gb300.solver import Solver
        s2 = Solver(p, 3, 3, 4, x, Ma=0.1, Re=400.0)
        m2 = O.make_mesh(p, x, 3, 3, 4)
        assert_parity(s2.rhs(q), O.rhs(qo, m2, gas), qo, m2, gas)
