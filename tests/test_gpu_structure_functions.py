"""lb_structure_functions over row lengths: against plain torch, and at a cost per node that does not
depend on the row length (the kernel is bound by its FP64 instructions; a row of 33 nodes given to warps
of its own issued 64 lanes' worth, 1.94 times)."""
import time

import numpy as np
import pytest
import torch

from paper_1111_0905_gb300 import config, lb

pytestmark = pytest.mark.gpu


def _lattice(nx, ny, nz):
    w = config.boiling_cell(nx, nz=nz, ny=ny, precision=lb.LB_FP32)
    lat = lb.Lattice(w.params, *[torch.from_numpy(x).cuda() for x in w.fields()])
    lat.step(3)
    return lat


@pytest.mark.parametrize("nx,ny,nz", [(2, 2, 1), (7, 300, 3), (33, 40, 5), (255, 3, 4), (256, 5, 2), (257, 4, 3), (300, 2, 2)])
def test_against_plain_sums(lblib, cuda, nx, ny, nz):
    lat = _lattice(nx, ny, nz)
    rmax, lo, hi = min(nx, ny) - 1, 0, nz
    got = lat.structure_functions(rmax, lo, hi)
    _, u, T = lat.moments()
    lat.close()
    for name, v in (("uz", u[2][lo:hi]), ("T", T[lo:hi])):
        for k in (2, 4):
            ref = [0.5 * sum((np.mean((np.roll(v, -r, a) - v) ** k)) for a in (1, 2)) for r in range(1, rmax + 1)]
            # sums of positive terms: at most their number times 2^-53 off, and 4 roundings per term
            assert np.allclose(got[f"S{k}_{name}"], ref, rtol=(nx * ny * nz + 8) * 2.0 ** -53, atol=0.0)


def test_cost_per_node_does_not_depend_on_the_row_length(lblib, cuda):
    best = {}
    for nx, ny in ((64, 512), (33, 993), (48, 683), (97, 338)):
        lat = _lattice(nx, ny, 24)
        times = []
        for _ in range(8):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            lat.structure_functions(32, 0, 24)
            times.append(time.perf_counter() - t0)
        lat.close()
        best[nx] = min(times) / (nx * ny)
    for nx in best:
        assert best[nx] <= 1.3 * best[64], best
