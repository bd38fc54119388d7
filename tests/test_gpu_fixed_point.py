"""The block fixed-point form of the float64 residual (csrc/rhs_fix.cuh) where its rules change: elements
inside and outside the fixed-point range side by side, neighbours beyond the near and the far series of
the logarithmic means, vanishing velocities, and partly filled CTAs at every degree (p = 1 to 3 put
16, 4 and 2 elements in a CTA).  Bound: the float64 rounding bound of the other parity tests."""
import numpy as np
import pytest
import torch

from oracle import esdc_oracle as O
from tests.gpu_common import assert_parity, geometry_rounding, make_pair

pytestmark = pytest.mark.gpu


def _case(p, kind, k=(3, 3, 3), flux="esc"):
    solver, q, mesh, gas, qo = make_pair(p, k, warp=0.1, seed=2, Re=400.0, Ma=0.4, volume_flux=flux)
    rng = np.random.default_rng(7 * p)
    x = qo.numpy().copy()
    rho, mom = x[:, 0], x[:, 1:4]
    pr = 0.4 * (x[:, 4] - 0.5 * (mom ** 2).sum(1) / rho)
    u = mom / rho[:, None]
    if kind == "far":                                    # up to 25% between neighbours: far series
        f = 1.0 + 0.12 * rng.uniform(-1, 1, rho.shape)
        g = 1.0 + 0.12 * rng.uniform(-1, 1, rho.shape)
    elif kind == "log":                                  # up to a factor of 4: logarithms, still in range
        f, g = 2.0 ** rng.uniform(-1, 1, rho.shape), 2.0 ** rng.uniform(-0.5, 0.5, rho.shape)
    elif kind == "range":                                # every fourth element outside the range
        f, g = np.ones_like(rho), np.ones_like(rho)
        f[::4] = 10.0 ** rng.uniform(-1.5, 1.5, f[::4].shape)
        g[1::8] = 10.0 ** rng.uniform(-1, 1, g[1::8].shape)
    else:                                                # "still": no velocity in most elements, tiny in the others
        f, g = 1.0 + 1e-3 * rng.uniform(-1, 1, rho.shape), np.ones_like(rho)
        u = u * np.where(np.arange(u.shape[0]) % 3 == 0, 1e-9, 0.0)[:, None, None, None, None]
    rho, pr = rho * f, pr * g
    x[:, 0], x[:, 1:4] = rho, rho[:, None] * u
    x[:, 4] = pr / 0.4 + 0.5 * rho * (u ** 2).sum(1)
    return solver, solver.to_device(x), mesh, gas, torch.tensor(x)


@pytest.mark.parametrize("kind", ["far", "log", "range", "still"])
@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 7])
def test_residual_parity_across_the_rules(p, kind):
    solver, q, mesh, gas, qo = _case(p, kind)
    assert_parity(solver.rhs(q), O.rhs(qo, mesh, gas), qo, mesh, gas)


@pytest.mark.parametrize("kind", ["log", "range", "still"])
@pytest.mark.parametrize("flux", ["kg", "dc"])
@pytest.mark.parametrize("p", [1, 2, 4, 5, 6, 7])
def test_variant_parity_across_the_rules(p, flux, kind):
    solver, q, mesh, gas, qo = _case(p, kind, flux=flux)
    assert_parity(solver.rhs(q), O.rhs(qo, mesh, gas, scheme=flux), qo, mesh, gas)


@pytest.mark.parametrize("kind", ["far", "range"])
@pytest.mark.parametrize("p,k", [(1, (11, 10, 9)), (2, (9, 8, 9)), (3, (7, 7, 7)), (4, (5, 6, 6)), (6, (5, 6, 6))])
def test_residual_parity_beyond_the_wide_form(p, k, kind):
    """Up to 1 to 6 elements per SM (by degree) run one element per CTA on more warps; these do not."""
    solver, q, mesh, gas, qo = _case(p, kind, k)
    assert_parity(solver.rhs(q), O.rhs(qo, mesh, gas), qo, mesh, gas)


@pytest.mark.parametrize("p", [1, 3, 7])
def test_nonphysical_state_stays_in_its_neighbourhood(p):
    """A node with negative pressure or a NaN takes its element and the neighbours that read it out of
    the fixed-point range, with the elements of their CTAs; what those hand on (their viscous traces)
    reaches one more ring, and every other element is unchanged."""
    solver, q, mesh, gas, qo = make_pair(p, (7, 5, 5), warp=0.05, seed=1)
    r = solver.rhs(q)
    bad = q.clone()
    bad[0, 4, 0, 0, 0] = -1.0
    bad[0, 0, -1, -1, -1] = float("nan")
    rb = solver.rhs(bad)
    epb = {1: 16, 3: 2, 7: 1}[p]
    near = {0} | {int(n) for n in mesh.nbr[0]}
    near = {k for e in near for k in range(e // epb * epb, min(q.shape[0], (e // epb + 1) * epb))}
    near |= {int(n) for e in near for n in mesh.nbr[e]}
    clean = [e for e in range(q.shape[0]) if e not in near]
    assert clean
    assert torch.isnan(rb[0]).any()
    assert torch.equal(rb[clean], r[clean])


@pytest.mark.parametrize("kind", ["far", "log", "range"])
@pytest.mark.parametrize("flux", ["esc", "kg"])
def test_p15_parity_across_the_rules(flux, kind):
    """p = 15 decides the range plane by plane."""
    solver, q, mesh, gas, qo = _case(15, kind, (2, 2, 1), flux)
    assert_parity(solver.rhs(q), O.rhs(qo, mesh, gas, scheme=flux), qo, mesh, gas, geo_rel=geometry_rounding(15))


@pytest.mark.parametrize("scale", [2.0 ** -60, 2.0 ** -43, 1.0, 2.0 ** 44, 2.0 ** 60])
def test_budget_logarithms(scale):
    """Entropy budgets with densities and pressures inside and beyond the exponents of the fixed-point
    logarithm.  Bound: 1e-13 of the terms' magnitudes, as in the other budget tests (the two sides build J
    independently), those of s = ln p - gamma ln rho taken before they cancel."""
    solver, q, mesh, gas, qo = make_pair(3, (3, 2, 2), warp=0.1, seed=3, Re=100.0)
    x = qo * scale
    d = torch.tensor(np.random.default_rng(1).uniform(-1, 1, tuple(x.shape))) * scale
    b, bo = solver.budgets(solver.to_device(x.numpy()), solver.to_device(d.numpy())), O.budgets(x, d, mesh, gas)
    PJ, g = O.quadrature_weights(mesh), gas.gamma
    rho, p = x[:, 0], (g - 1) * (x[:, 4] - 0.5 * (x[:, 1:4] ** 2).sum(1) / x[:, 0])
    logs = (p.log().abs() + g * rho.log().abs() + g) / (g - 1)
    wd = logs * d[:, 0].abs() + rho / p * ((x[:, 1:4] * d[:, 1:4]).abs().sum(1) / rho + d[:, 4].abs()
                                          + 0.5 * (x[:, 1:4] ** 2).sum(1) / rho ** 2 * d[:, 0].abs())
    eps = 1e-13
    assert abs(b[0] - bo[0]) <= eps * float((PJ * rho * logs).sum())
    assert abs(b[1] - bo[1]) <= eps * abs(bo[1])
    assert abs(b[2] - bo[2]) <= eps * float((PJ * wd).sum())
