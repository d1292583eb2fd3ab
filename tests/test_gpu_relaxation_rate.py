"""The relaxation rate that an FP32 context gets is its tau's to single precision.

In a uniform state at rest, f and g carry in addition a mode without density, momentum or energy,
+A on the diagonals (1, 1, 0), (-1, -1, 0) and -A on (1, -1, 0), (-1, 1, 0). Streaming leaves it, the
equilibria and the force do not see it, so n steps multiply it by (1 - 1/tau)^n exactly. In single
precision each step may round the factor and the product (2^-24 each, relative) and the state is
rounded once at the start: (2 n + 1) 2^-24 in all. At tau = 1 nothing is left of the mode but the
rounding of the double-precision export (1e-17)."""
import numpy as np
import pytest

from paper_1111_0905_gb300 import lb

pytestmark = pytest.mark.gpu

A = 1e-3


@pytest.mark.parametrize("shape", [(7, 6, 5), (96, 96, 96)])     # three kernels; march
@pytest.mark.parametrize("tau", [0.502, 0.505, 0.51, 0.6, 0.7, 0.8, 0.9, 1.0, 1.25, 2.0, 4.0])
def test_fp32_relaxation_rate(lblib, cuda, shape, tau):
    nx, ny, nz = shape
    p = lb.Params(nx, ny, nz, tau_nu=tau, tau_kappa=tau, G=-2.0, kappa=0.5 * (tau - 0.5), T_d=1.0 / 3.0, T_u=1.0 / 3.0,
                  rho0=1.5, T0=1.0 / 3.0, precision=lb.LB_FP32)
    rho = np.full((nz, ny, nx), 1.5)
    lat = lb.Lattice(p, rho, np.full((nz, ny, nx), 1.0 / 3.0))
    # the rest equilibria at the reference state, whose stored deviations are 0 (lb_init's differ by the
    # rounding of rho T in single precision, 1e-8)
    csq = np.array([0] + [1] * 6 + [2] * 12).reshape(19, 1, 1, 1)
    w = np.array([1 / 3, 1 / 18, 1 / 36])[csq]
    lam = p.kappa / (p.c_v * (tau - 0.5))     # = rho T: well inside the window of g's equilibrium
    T0 = 1.0 / 3.0
    base = [b * np.ones((nz, ny, nx)) for b in (w * 1.5, w * (1.5 * T0 + 4.5 * (lam * T0 - 0.5 * T0) * (csq - 1)))]
    mode = np.zeros((19, 1, 1, 1))
    mode[7:9], mode[9:11] = A, -A
    lat.set_populations(*[np.ascontiguousarray(b + mode) for b in base])
    factor = 1.0 - 1.0 / tau
    # as many steps as leave a hundredth of the mode, 64 at most
    n = 1 if factor == 0.0 else min(64, max(1, int(np.log(1e-2) / np.log(abs(factor)))))
    lat.step(n)
    after = lat.populations()
    lat.close()
    expect = mode * factor ** n
    tol = 1e-15 if factor == 0.0 else (2 * n + 1) * 2.0 ** -24 * A * abs(factor) ** n
    for b, x in zip(base, after):
        err = np.abs((x - b) - expect)[7:11].max()
        assert err <= tol, (tau, n, err / tol)
