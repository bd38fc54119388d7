"""The ES-C adjoint where its rules change (csrc/adj_pairs_fix.cu): neighbours beyond the near and the far series
of the logarithmic means, elements outside the fixed-point range beside others in partly filled CTAs (p = 1 to 3 put
16, 4 and 2 elements in one), cotangents far from one, non-finite ones, and zero.  Against the oracle's autograd with
the tolerance of the other adjoint tests, 1e-10 normwise."""
import pytest
import torch

from oracle import esdc_oracle as O
from tests.gpu_common import EPS64, make_pair, normwise_errors
from tests.test_gpu_fixed_point import _case

pytestmark = pytest.mark.gpu


def _lam(qo, seed=11):
    return torch.randn(qo.shape, generator=torch.Generator().manual_seed(seed), dtype=torch.float64)


@pytest.mark.parametrize("kind", ["far", "log", "range"])
@pytest.mark.parametrize("p,k", [(1, (3, 3, 3)), (2, (3, 3, 1)), (3, (3, 3, 3)), (4, (3, 2, 2)), (5, (3, 2, 2)), (6, (3, 2, 2)), (7, (3, 2, 1))])
def test_vjp_across_the_rules(p, k, kind):
    solver, q, mesh, gas, qo = _case(p, kind, k)
    lam = _lam(qo)
    qq = qo.clone().requires_grad_(True)
    (go,) = torch.autograd.grad(O.rhs(qq, mesh, gas), qq, lam)
    e = normwise_errors(solver.rhs_vjp(q, lam.cuda()), go)
    print("vjp", kind, ["%.1e" % x for x in e])
    assert max(e) <= 1e-10, e


@pytest.mark.parametrize("scale", [2.0 ** -300, 2.0 ** -80, 2.0 ** 80, 2.0 ** 300])
@pytest.mark.parametrize("p", [2, 4, 7])
def test_cotangents_far_from_one(p, scale):
    """The gradient is linear in the cotangent, inside and outside the fixed-point range of its exponents."""
    solver, q, mesh, gas, qo = _case(p, "far", (3, 2, 2))
    lam = _lam(qo).cuda()
    g = solver.rhs_vjp(q, lam)
    gs = solver.rhs_vjp(q, lam * scale) / scale
    assert max(normwise_errors(gs, g.cpu())) <= 1e-10
    assert float(solver.rhs_vjp(q, torch.zeros_like(lam)).abs().max()) == 0.0


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("p", [1, 3, 7])
def test_nonfinite_cotangent_stays_in_its_neighbourhood(p, bad):
    """A non-finite cotangent at one node reaches its element and, by the faces and the viscous lift, two rings of
    neighbours; every other gradient is unchanged but for the elements of the same CTAs, which change form."""
    solver, q, mesh, gas, qo = _case(p, "far", (7, 5, 5))
    lam = _lam(qo).cuda()
    g = solver.rhs_vjp(q, lam)
    lb = lam.clone()
    lb[0, 2, 0, 0, 0] = bad
    gb = solver.rhs_vjp(q, lb)
    near = {0}
    for _ in range(2):
        near |= {int(n) for e in near for n in mesh.nbr[e]}
    same = [e for e in range(q.shape[0]) if e not in near]
    assert not torch.isfinite(gb[0]).all()
    assert torch.isfinite(gb[same]).all()
    assert max(normwise_errors(gb[same], g[same].cpu())) <= 1e-10


@pytest.mark.parametrize("p", [2, 3, 4, 5, 6, 7])
def test_one_large_cotangent_leaves_other_lines_alone(p):
    """Inviscid, without dissipation, the gradient at an element's interior nodes takes the cotangents of its three
    lines only: one of 1e10 at a corner node, on none of them, must not cost it bits.  Bound: 64 N eps of the largest
    interior value (3 N pair terms of about ten roundings), a hundred times that for density and energy (differences
    of pressure terms)."""
    solver, qg, mesh, gas, qo = make_pair(p, (3, 2, 2), warp=0.1, seed=3, Re=0.0, dissipation=False, noise=2e-2)
    lam = _lam(qo).cuda()
    g = solver.rhs_vjp(qg, lam)
    big = lam.clone()
    big[:, :, 0, 0, 0] = 1e10
    inner = (slice(None), slice(None)) + (slice(1, -1),) * 3
    e = normwise_errors(solver.rhs_vjp(qg, big)[inner], g[inner].cpu())
    print("interior", ["%.1e" % x for x in e])
    assert max(e[1:4]) <= 64 * (p + 1) * EPS64, e
    assert max(e) <= 6400 * (p + 1) * EPS64, e
