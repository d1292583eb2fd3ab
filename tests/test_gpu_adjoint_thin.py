"""The adjoint on cells of one or two planes, columns or rows, where a plane is both walls at once and a
node its own neighbour: against the oracle's gradient, as test_gpu_adjoint.py does."""
import numpy as np
import pytest

from paper_1111_0905_gb300 import config, lb
from test_gpu_adjoint import _oracle_grad

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(6, 5, 1), (7, 1, 2), (1, 6, 4), (2, 2, 3), (1, 1, 1), (1, 1, 5), (130, 2, 2)])
@pytest.mark.parametrize("prec", [lb.LB_FP64, lb.LB_FP32])
def test_adjoint_of_thin_cells(lblib, cuda, shape, prec):
    nx, ny, nz = shape
    w = config.boiling_cell(nx, nz=nz, ny=ny, precision=prec)
    rho, T = w.fields()
    lat = lb.Lattice(w.params, rho, T)
    got = lat.adjoint(6, 4, grad_T0=True)
    lat.close()
    ref = _oracle_grad(w.params, rho, T, 6)
    tol_J, tol = (1e-11, 1e-9) if prec == lb.LB_FP64 else (1e-5, 1e-4)
    assert abs(got["J"] - ref["J"]) <= tol_J * max(1.0, abs(ref["J"]))
    for k in ("T_d", "T_u", "G"):
        assert abs(got[k] - ref[k]) <= tol * max(1.0, abs(ref[k])), (k, got[k], ref[k])
    assert np.abs(got["T0"] - ref["T0"]).max() <= tol * np.abs(ref["T0"]).max()
