"""FP32 compute over the densities that single precision holds: a uniform state at rest has T = E/rho.

1/rho of a density above 2^126 is a subnormal number, not 0. Bound: 1/rho is within 2^-24 of itself (of
the subnormal spacing, 1.4e-45, above 2^126), E and the product round once each: 2^-22 covers them."""
import numpy as np
import pytest

from paper_1111_0905_gb300 import lb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(7, 6, 5), (96, 96, 96)])     # three kernels; march
@pytest.mark.parametrize("rho", [1e-30, 1.0, 1.7, 1e30, 8.6e37, 1.2e38])
def test_temperature_of_a_uniform_state(lblib, cuda, shape, rho):
    nx, ny, nz = shape
    T = 1.0 / 3.0
    p = lb.Params(nx, ny, nz, tau_nu=1.0, tau_kappa=1.0, G=-2.0, kappa=0.1 * rho, T_d=T, T_u=T, rho0=rho, T0=T,
                  precision=lb.LB_FP32)
    lat = lb.Lattice(p, np.full((nz, ny, nx), rho), np.full((nz, ny, nx), T))
    r, u, t = lat.moments()
    lat.close()
    assert np.abs(r / rho - 1.0).max() <= 2.0 ** -22
    assert np.abs(t / T - 1.0).max() <= 2.0 ** -22
    assert all(np.abs(x).max() <= 1e-12 for x in u)
