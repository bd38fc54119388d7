"""Supersonic flow along one axis, where the transverse momentum fluxes are far smaller than the kinetic part along
the axis: they keep the bits that float64 gives them.  Bound: the float64 rounding bound of the other parity tests
(which leaves out the rounding of the pressure as a difference of energies, larger from Mach 6 on)."""
import pytest

from oracle import esdc_oracle as O
from tests.gpu_common import assert_parity
from tests.test_gpu_stretched import _pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flow", ["x", "z", "all"])
@pytest.mark.parametrize("flux", ["esc", "kg", "dc"])
@pytest.mark.parametrize("p,Ma,Re", [(5, 6.0, 0.0), (7, 2.0, 0.0), (7, 2.0, 500.0), (7, 4.0, 0.0)])
def test_residual_parity(p, Ma, Re, flux, flow):
    solver, q, mesh, gas, qo = _pair(p, 1.0, flow, flux, Re=Re, Ma=Ma)
    assert_parity(solver.rhs(q), O.rhs(qo, mesh, gas, scheme=flux), qo, mesh, gas)
