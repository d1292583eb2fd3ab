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


@pytest.mark.parametrize("shape", [(16, 9, 10), (96, 96, 96)])     # three kernels; march
@pytest.mark.parametrize("rho0", [0.005, 0.013, 0.015, 0.02, 0.03, 1.5, 40.0])
def test_force_at_a_distant_reference_density(lblib, cuda, shape, rho0):
    """The reference density of the deviations is the caller's choice. The velocity that the force gives a
    state at rest, against the FP64 form: psi = psi(rho0) e^t, t = 1/rho0 - 1/rho <= 77 (200 where the
    reference is set apart from it), is good to
    77 2^-23 from the rounding of t and 92 2^-23 from the fast exponential (2 + 1.16 |t| ulp), 2e-5; the
    weighted sum of neighbours (weights adding up to 1, psi <= 0.6) then to 1.2e-5 of its largest value,
    0.05 for the wave below, 2.4e-4 relative."""
    nx, ny, nz = shape
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    rho = 1.5 * (1.0 + 0.2 * np.cos(2.0 * np.pi * x / 8.0)) * np.ones(shape[::-1])
    T = np.full(shape[::-1], 1.0 / 3.0)
    out = []
    for prec in (lb.LB_FP64, lb.LB_FP32):
        p = lb.Params(nx, ny, nz, tau_nu=1.0, tau_kappa=1.0, G=-2.7, kappa=0.1, T_d=1.0 / 3.0, T_u=1.0 / 3.0, rho0=rho0,
                      T0=1.0 / 3.0, precision=prec)
        lat = lb.Lattice(p, rho, T)
        out.append(np.stack(lat.moments()[1]))
        lat.close()
    scale = np.abs(out[0]).max()
    assert scale > 0.01
    assert np.abs(out[1] - out[0]).max() <= 5e-4 * scale
