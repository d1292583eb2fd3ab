"""Looking at a run does not change it: the populations are the same bit for bit whether steps take Nu
samples or not, whether lb_nusselt, lb_diagnostics, a health check or lb_save comes between them, and
after lb_load. On cells that step in every form that the library chooses: three kernels, the march, the
march with two nodes per thread (16-bit deviations, even nx)."""
import pytest
import torch

from paper_1111_0905_gb300 import config, lb

pytestmark = pytest.mark.gpu

SMALL = (20, 14, 9)
CELLS = [("f64", SMALL), ("f32", SMALL), ("f32", (96, 96, 96)), ("fp16loc", SMALL), ("fp16loc", (159, 104, 64))]
CELLS += [(prec, cell) for prec in ("fp16dev", "bf16dev")
          for cell in (SMALL, (127, 119, 77), (128, 98, 96), (64, 200, 121), (256, 256, 4))]


def _lattice(prec, cell, **kw):
    nx, ny, nz = cell
    w = config.boiling_cell(nx, nz=nz, ny=ny, precision=lb.PRECISIONS[prec], kappa=0.15, tau_nu=1.25)
    rho, T = w.fields()
    p = lb.Params(**{**w.params.__dict__, **kw})
    return lb.Lattice(p, torch.from_numpy(rho).cuda(), torch.from_numpy(T).cuda())


def _state(lat):
    f, g = lat.populations(device=True)
    lat.close()
    return f, g


def _equal(a, b):
    return torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("prec,cell", CELLS)
def test_looking_does_not_change_the_run(lblib, cuda, tmp_path, prec, cell):
    lat = _lattice(prec, cell)
    lat.step(8)
    plain = _state(lat)
    # every step samples; every second one; with a health check in between
    for opts in ({"nu_every": 1}, {"nu_every": 2}, {"nu_every": 2, "check_every": 3}):
        lat = _lattice(prec, cell, **opts)
        lat.step(8)
        avg = lat.nusselt()[2]
        assert _equal(_state(lat), plain), opts
        # the samples that a sampling step takes in passing are those of separate moments passes
        lat = _lattice(prec, cell, **opts)
        for _ in range(8):
            lat.step(1)
            lat.nusselt()
            lat.diagnostics()
        assert abs(lat.nusselt()[2] - avg) <= 1e-4 * max(1.0, abs(avg)), opts
        assert _equal(_state(lat), plain), opts
    # saved at a due sample, and taken up again
    lat = _lattice(prec, cell, nu_every=2)
    lat.step(4)
    lat.save(tmp_path / "state")
    lat.step(4)
    assert _equal(_state(lat), plain)
    lat = _lattice(prec, cell)
    lat.load(tmp_path / "state")
    lat.step(4)
    assert _equal(_state(lat), plain)
