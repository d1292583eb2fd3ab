"""lb_step_info names the kernel that lb_step launches: the form, its grid over the cell, its threads. And
parity with the oracle at full size on the seams of that kernel: the tiles and the z chunks of its own
grid (test_gpu_fullsize.py samples those of the tile march)."""
import numpy as np
import pytest
import torch

from helpers import oracle_cutout_moments
from paper_1111_0905_gb300 import config, lb

pytestmark = pytest.mark.gpu

# threads per CTA and tile of each form: the ring's threads (rounded up to warps) and the tile's
MARCH = {"f32": (448 + 256, 32, 8), "fp16dev": (448 + 256, 32, 8), "bf16dev": (448 + 256, 32, 8),
         "fp16loc": (416 + 224, 32, 7)}
MARCH2 = (384 + 224, 64, 7)


def step_info(prec, nx, ny, nz, **kw):
    w = config.boiling_cell(nx, nz=nz, ny=ny, precision=lb.PRECISIONS[prec])
    p = lb.Params(**{**w.params.__dict__, **kw})
    lat = lb.Lattice(p, *[torch.from_numpy(x).cuda() for x in w.fields()])
    info, tile = lat.step_info(), lat.launch_info()
    lat.close()
    return info, tile


@pytest.mark.parametrize("prec,cell,form", [
    ("f64", (24, 24, 24), "three kernels"), ("f64", (96, 96, 96), "three kernels"), ("f32", (24, 24, 24), "three kernels"),
    ("f32", (96, 96, 96), "march"), ("fp16loc", (159, 104, 64), "march"), ("fp16dev", (127, 119, 77), "march"),
    ("fp16dev", (128, 98, 96), "march, two nodes per thread"), ("bf16dev", (64, 200, 121), "march, two nodes per thread")])
def test_form_and_shape(lblib, cuda, prec, cell, form):
    info, _ = step_info(prec, *cell)
    nx, ny, nz = cell
    assert info["form"] == form
    if form == "three kernels":
        assert info["threads_per_cta"] in (32, 64, 256)
        assert info["grid"] == [-(-nx * ny // info["threads_per_cta"]), nz] and info["smem_bytes"] == 0
    else:
        threads, tx, ty = MARCH2 if "two" in form else MARCH[prec]
        assert info["threads_per_cta"] == threads and info["ctas_per_sm"] == 1
        assert info["grid"][0] == -(-nx // tx) * -(-ny // ty) and 1 <= info["grid"][1] <= nz
        assert info["threads_per_cta"] * info["registers"] <= 65536 and info["smem_bytes"] > 0
    assert info["registers"] > 0


def test_a_given_launch_shape_is_the_tile_march(lblib, cuda):
    for kw in ({"tile_y": 8}, {"z_chunk": 12}):
        info, tile = step_info("f32", 96, 96, 96, **kw)
        assert info["form"] == "tile march"
        assert {k: info[k] for k in tile} == tile


def test_variants_have_no_two_node_march(lblib, cuda):
    info, _ = step_info("fp16dev", 128, 98, 96, forcing=lb.LB_FORCE_GUO)
    assert info["form"] != "march, two nodes per thread"


def _seam_nodes(p, tx, ty, zc, seed):
    nx, ny, nz = p.nx, p.ny, p.nz
    xs = [0, tx - 1, tx, nx // tx // 2 * tx, nx - 1]
    ys = [0, ty - 1, ty, ny // ty // 2 * ty, ny - 1]
    zs = sorted({z for c in range(0, nz, zc) for z in (c - 1, c, c + 1) if 0 <= z < nz} | {nz - 1})
    rng = np.random.default_rng(seed)
    pick = rng.permutation(len(zs))[:16]
    return [(xs[k % 5], ys[(k // 2) % 5], zs[i]) for k, i in enumerate(pick)]


CELLS = [("single", 128, "f32", 1e-5, 1e-5), ("boiling", 256, "bf16dev", 2e-3, None), ("boiling", 256, "fp16loc", 2e-3, None),
         ("boiling", 512, "f32", 1e-5, 1e-5), ("boiling", 512, "fp16dev", 2e-3, None), ("boiling", 512, "fp16loc", 2e-3, None)]


@pytest.mark.parametrize("cell,n,prec,tol,tol_u", CELLS)
def test_full_size_parity_on_the_seams(lblib, cuda, cell, n, prec, tol, tol_u):
    make = config.single_phase_cell if cell == "single" else config.paper_scale_cell
    w = make(n, precision=lb.PRECISIONS[prec])
    p = w.params
    rho, T = w.fields()
    lat = lb.Lattice(p, torch.from_numpy(rho).cuda(), torch.from_numpy(T).cuda())
    info = lat.step_info()
    assert info["form"].startswith("march")
    _, tx, ty = MARCH2 if "two" in info["form"] else MARCH[prec]
    lat.step(2)
    r, u, t = lat.moments(device=True)
    nodes = _seam_nodes(p, tx, ty, -(-p.nz // info["grid"][1]), n)
    idx = torch.tensor([(z * p.ny + y) * p.nx + x for x, y, z in nodes], device="cuda")
    gpu = torch.stack([v.reshape(-1)[idx] for v in (r, *u, t)], dim=1).cpu().numpy()
    lat.close()
    ora = oracle_cutout_moments(p, rho, T, 2, nodes)
    for k in (0, 4):
        assert np.abs(gpu[:, k] - ora[:, k]).max() < tol * np.abs(ora[:, k]).max()
    if tol_u is not None:
        assert np.abs(gpu[:, 1:4] - ora[:, 1:4]).max() < tol_u * max(np.abs(ora[:, 1:4]).max(), 1e-2)
