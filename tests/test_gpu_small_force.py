"""The force of the FP32 three-kernel step is the one that the velocity pass formed, not one recovered from
the rounded velocity: a state in uniform fast motion under a small gravity gains rho g_z a step, to the
roundings of its populations. Away from the walls one step changes j by F whole (the velocity shift and
Guo forcing alike). Its error over many velocities is compared with the tile march's, which keeps F: both
round their populations alike, while half a unit in the last place of u, 2^-25 |u|, times 2 rho would
come on top (several times the rest)."""
import numpy as np
import pytest

from paper_1111_0905_gb300 import lb

pytestmark = pytest.mark.gpu

C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
              (0, -1, 1)])
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


@pytest.mark.parametrize("forcing", [lb.LB_FORCE_SHIFT, lb.LB_FORCE_GUO])
@pytest.mark.parametrize("tau", [1.0, 5.0])
def test_momentum_gain_of_a_moving_state(lblib, cuda, forcing, tau):
    nx, ny, nz, rho, T, gz = 4, 4, 16, 1.5, 1.0 / 3.0, -1e-8
    velocities = np.random.default_rng(3).uniform(-0.12, 0.12, (200, 3))
    errors = {}
    for tile_y in (0, 8):
        p = lb.Params(nx, ny, nz, tau_nu=tau, tau_kappa=1.0, G=-2.0, kappa=0.2, g_z=gz, T_d=T, T_u=T, rho0=rho, T0=T,
                      precision=lb.LB_FP32, forcing=forcing, tile_y=tile_y)
        lat = lb.Lattice(p, np.full((nz, ny, nx), rho), np.full((nz, ny, nx), T))
        assert lat.step_info()["form"] == ("tile march" if tile_y else "three kernels")
        err = []
        for u in velocities:
            cu, uu = C @ u, u @ u
            k = (C ** 2).sum(1) - 1
            e = 1.0 + 3.0 * cu + 4.5 * cu ** 2 - 1.5 * uu
            feq = W * rho * (e + 4.5 * k * (T - 1 / 3))
            geq = W * (rho * T * e + 4.5 * k * (0.4 * T - rho * T / 3))       # lam = kappa/(c_v (tau_kappa - 1/2))
            lat.set_populations(*[np.ascontiguousarray(np.broadcast_to(q[:, None, None, None], (19, nz, ny, nx)))
                                  for q in (feq, geq)])
            j0 = np.tensordot(C.T, lat.populations()[0], 1)[:, nz // 2]
            lat.step(1)
            j1 = np.tensordot(C.T, lat.populations()[0], 1)[:, nz // 2]
            err.append((j1 - j0 - np.array([0.0, 0.0, rho * gz])[:, None, None]).ravel())
        lat.close()
        errors[tile_y] = float(np.sqrt(np.mean(np.square(err))))
    assert errors[0] <= 1.5 * errors[8], errors
