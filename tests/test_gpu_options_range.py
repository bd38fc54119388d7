"""The optional interface terms (matrix dissipation, interior penalty, surface metrics of the optimized metrics,
bounded boxes with exterior data and a source) in elements outside the fixed-point range beside others inside it,
and in boxes of stretched elements, which take the float64 kernel.  Bound: the float64 rounding bound of the other
parity tests."""
import numpy as np
import pytest
import torch

from oracle import esdc_oracle as O
from paper_1911_10966_gb300 import inputs as I
from tests.gpu_common import assert_parity, make_pair
from tests.test_gpu_mms import _pair

pytestmark = pytest.mark.gpu


def _out_of_range(q, seed):
    """Every fourth element's density and every eighth's pressure scattered over one to three decades."""
    x, rng = np.asarray(q).copy(), np.random.default_rng(seed)
    rho, mom = x[:, 0].copy(), x[:, 1:4].copy()
    pr = 0.4 * (x[:, 4] - 0.5 * (mom ** 2).sum(1) / rho)
    f, g = np.ones_like(rho), np.ones_like(rho)
    f[::4] = 10.0 ** rng.uniform(-1.5, 1.5, f[::4].shape)
    g[1::8] = 10.0 ** rng.uniform(-1, 1, g[1::8].shape)
    x[:, 0], x[:, 1:4] = rho * f, mom * f[:, None]
    x[:, 4] = pr * f * g / 0.4 + 0.5 * x[:, 0] * ((mom / rho[:, None]) ** 2).sum(1)
    return x


OPTIONS = [("curl", {"dissipation": "matrix", "ip_coef": 2.0}), ("optimized", {}),
           ("optimized", {"dissipation": "matrix", "ip_coef": 1.0}), ("curl", {"ip_coef": 1.0})]


@pytest.mark.parametrize("vf", ["esc", "kg", "dc"])
@pytest.mark.parametrize("metrics,kw", OPTIONS)
@pytest.mark.parametrize("p,k", [(1, (3, 3, 3)), (2, (3, 3, 2)), (3, (3, 2, 2)), (5, (2, 2, 2)), (7, (2, 2, 2))])
def test_out_of_range_parity(p, k, metrics, kw, vf):
    from paper_1911_10966_gb300.solver import Solver
    s0, qg, mesh, gas, qo = make_pair(p, k, warp=0.1, seed=5, Re=400.0, noise=2e-2, volume_flux=vf, metrics=metrics)
    solver = Solver(p, *k, s0.coords, Re=400.0, volume_flux=vf, metrics=metrics, **kw)
    x = _out_of_range(qo.numpy(), p)
    qo = torch.tensor(x)
    ro = O.rhs(qo, mesh, gas, dissipation=kw.get("dissipation", True), scheme=vf, ip_coef=kw.get("ip_coef", 0.0))
    assert_parity(solver.rhs(solver.to_device(x)), ro, qo, mesh, gas)


@pytest.mark.parametrize("vf", ["esc", "kg", "dc"])
@pytest.mark.parametrize("metrics,kw", OPTIONS)
@pytest.mark.parametrize("p,k", [(1, (3, 3, 3)), (3, (3, 2, 2)), (6, (2, 2, 2))])
def test_stretched_parity(p, k, metrics, kw, vf):
    from paper_1911_10966_gb300.solver import Solver
    box = ([0.0] * 3, [1.0, 1.0, 8.0])
    s0, qg, mesh, gas, qo = make_pair(p, k, warp=0.05, seed=5, Re=400.0, noise=2e-2, volume_flux=vf, metrics=metrics, box=box)
    solver = Solver(p, *k, s0.coords, Re=400.0, volume_flux=vf, metrics=metrics, lo=box[0], hi=box[1], **kw)
    ro = O.rhs(qo, mesh, gas, dissipation=kw.get("dissipation", True), scheme=vf, ip_coef=kw.get("ip_coef", 0.0))
    assert_parity(solver.rhs(qg), ro, qo, mesh, gas)


@pytest.mark.parametrize("p,k,kw", [(1, 3, {}), (2, 3, {"dissipation": "matrix", "ip_coef": 2.0}), (3, 2, {"volume_flux": "kg"}),
                                    (4, 2, {"volume_flux": "dc"}), (7, 2, {})])
def test_bounded_out_of_range_parity(p, k, kw):
    solver, xg, mesh, xo, gas = _pair(p, k, 0.1, 4.0e2, **kw)
    x = _out_of_range(I.perturb(I.manufactured(xo), seed=4, rel=1e-2), p)
    src = I.random_direction(x.shape, seed=5, scale=1.0)
    ext, sg = solver.to_device(I.manufactured(xg)), solver.to_device(src)
    solver.set_exterior(ext)
    solver.set_source(sg)
    qo = torch.tensor(x)
    ro = O.rhs(qo, mesh, gas, dissipation=kw.get("dissipation", True), scheme=kw.get("volume_flux", "esc"),
               ip_coef=kw.get("ip_coef", 0.0), q_ext=torch.tensor(I.manufactured(xo)), source=torch.tensor(src))
    assert_parity(solver.rhs(solver.to_device(x)), ro, qo, mesh, gas)
