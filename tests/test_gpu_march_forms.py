"""The marches on cells that take them, the form asserted through lb_step_info: against the tile march
(tile_y = 8, itself pinned to the oracle), with the tolerances of test_gpu_step_forms.py, and against
themselves with other chunks and tiles."""
import pytest
import torch

from paper_1111_0905_gb300 import config, lb
from test_gpu_step_forms import _cell, _same

pytestmark = pytest.mark.gpu

ONE, TWO = "march", "march, two nodes per thread"
# narrower than a tile and its ring (periodic wrap inside it); a tile with one column or row; one short of
# a tile; chunks of four planes and uneven last ones; 4 planes in all
F32 = [(31, 193, 30), (161, 39, 44), (98, 135, 80), (127, 119, 77), (608, 62, 4), (24, 400, 96)]
# tiles of 7 rows, windows of references: as above, and 3 and 6 chunks
LOC = [(31, 264, 84), (641, 49, 30), (64, 169, 63), (32, 209, 85), (160, 35, 108), (255, 132, 16), (159, 104, 64)]
# tiles of 64 x 7: one pair in the last tile, one pair short of it, narrower than a tile, one row, six rows
PAIR = [(322, 35, 30), (62, 42, 100), (126, 33, 72), (114, 99, 30), (64, 41, 100), (246, 263, 4), (192, 203, 96)]
ODD = [(127, 119, 77), (31, 1200, 64)]


def _form(p, rho, T):
    lat = lb.Lattice(p, rho, T)
    info = lat.step_info()
    lat.close()
    return info


@pytest.mark.parametrize("prec,cell,form",
                         [("f32", c, ONE) for c in F32] + [("fp16loc", c, ONE) for c in LOC]
                         + [(q, c, TWO) for q in ("fp16dev", "bf16dev") for c in PAIR]
                         + [(q, c, ONE) for q in ("fp16dev", "bf16dev") for c in ODD])
@pytest.mark.parametrize("nu_every", [1, 0])
def test_march_against_tile_march(lblib, cuda, prec, cell, form, nu_every):
    p, rho, T = _cell(prec, *cell, nu_every=nu_every)
    assert _form(p, rho, T)["form"] == form
    _same(prec, p, rho, T, 3)


@pytest.mark.parametrize("prec,cell", [("f32", (98, 135, 80)), ("f32", (31, 193, 30)), ("fp16loc", (64, 169, 63)),
                                       ("fp16loc", (159, 104, 64)), ("fp16dev", (127, 119, 77))])
@pytest.mark.parametrize("forcing,psi", [(1, 0), (0, 1), (1, 1)])
def test_variants_in_the_march(lblib, cuda, prec, cell, forcing, psi):
    p, rho, T = _cell(prec, *cell, forcing, psi)
    assert _form(p, rho, T)["form"] == ONE
    _same(prec, p, rho, T, 3)


@pytest.mark.parametrize("prec,cell,form", [("f32", (32, 40, 120), ONE), ("f32", (64, 40, 60), ONE),
                                            ("fp16loc", (64, 133, 60), ONE), ("fp16loc", (32, 133, 120), ONE),
                                            ("fp16dev", (64, 49, 84), TWO), ("bf16dev", (64, 49, 102), TWO)])
def test_result_does_not_depend_on_the_chunk(lblib, cuda, prec, cell, form):
    """A cell and the same cell repeated in y march in chunks of other lengths; bit for bit the same."""
    nx, ny, nz = cell
    w = config.boiling_cell(nx, nz=nz, ny=ny, precision=lb.PRECISIONS[prec], kappa=0.15, tau_nu=1.25)
    rho, T = (torch.from_numpy(x).cuda() for x in w.fields())
    out = []
    for k in (1, 2):
        p = lb.Params(**{**w.params.__dict__, "ny": k * ny, "rho0": w.rho_mean, "T0": 1.0 / 3.0})
        lat = lb.Lattice(p, torch.cat([rho] * k, dim=1).contiguous(), torch.cat([T] * k, dim=1).contiguous())
        info = lat.step_info()
        assert info["form"] == form
        lat.step(6)
        out.append((info["grid"][1], *lat.populations(device=True)))
        lat.close()
    assert out[0][0] != out[1][0]
    for a, b in zip(out[0][1:], out[1][1:]):
        assert torch.equal(torch.cat([a, a], dim=2), b)
