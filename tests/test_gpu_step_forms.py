"""The forms of the step against each other: a context that leaves its launch shape to the library
(three streaming kernels, or the march with separate warps for moments and collision) against the
tile march of the same cell (tile_y = 8, itself pinned to the oracle).

The forms differ in the order of sums and in contractions only, so per step they differ by a few
roundings of the compute precision. Tolerances, relative to the field's largest magnitude, are those
of the parity tests: FP64 1e-12 and FP32 1e-5 on populations, rho, T and (with their floors) u; 16-bit
2e-3 on populations, rho and T. No bound on u is asked of 16-bit storage: one rounding of a population
of magnitude 2^-5 that falls the other way moves j by 2^-13 (BF16), more than 1e-2 of the floor. Sizes: one node past and short
of a tile (32 x 8, 32 x 7, 64 x 7), a warp and a chunk, one pair of nodes in a tile; one and two planes; the smallest cells that march."""
import numpy as np
import pytest
import torch

from paper_1111_0905_gb300 import config, lb, synthetic

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 1e-5, "fp16loc": 2e-3, "fp16dev": 2e-3, "bf16dev": 2e-3}
U_FLOOR = {"f64": 1e-3, "f32": 1e-2}     # as in the parity tests: velocity rounding is absolute


def _cell(prec, nx, ny, nz, forcing=0, psi=0, **kw):
    w = config.boiling_cell(nx, nz=nz, ny=ny, precision=lb.PRECISIONS[prec], kappa=0.15, tau_nu=1.25)
    p = w.params
    p.forcing, p.psi_kind = forcing, psi
    for k, v in kw.items():
        setattr(p, k, v)
    rho, T = w.fields()
    if psi == lb.LB_PSI_VDW:
        rho, _ = synthetic.boiling_fields(nx, ny, nz, 3.5, p.T_d, p.T_u, 0.05)
    return p, torch.from_numpy(rho).cuda(), torch.from_numpy(T).cuda()


def _outputs(p, rho, T, steps, **kw):
    lat = lb.Lattice(lb.Params(**{**p.__dict__, **kw}), rho, T)
    lat.step(steps)
    f, g = lat.populations(device=True)
    r, u, t = lat.moments(device=True)
    nu = lat.nusselt()
    lat.close()
    return f, g, r, torch.stack(u), t, nu


def _rel(a, b, floor=0.0):
    return float((a - b).abs().max() / max(float(b.abs().max()), floor))


def _same(prec, p, rho, T, steps):
    a, b = _outputs(p, rho, T, steps), _outputs(p, rho, T, steps, tile_y=8)
    tol = TOL[prec]
    for x, y in zip((a[0], a[1], a[2], a[4]), (b[0], b[1], b[2], b[4])):
        assert _rel(x, y) <= tol
    if prec in U_FLOOR:
        assert _rel(a[3], b[3], U_FLOOR[prec]) <= tol
    assert np.abs(a[5][1] - b[5][1]).max() <= max(tol, 1e-9) * max(1.0, np.abs(b[5][1]).max())
    if p.nu_every:
        assert abs(a[5][2] - b[5][2]) <= max(tol, 1e-9) * max(1.0, abs(b[5][2]))
    # deterministic: the same run again, bit for bit
    c = _outputs(p, rho, T, steps)
    assert all(torch.equal(x, y) for x, y in zip(a[:5], c[:5])) and a[5][0] == c[5][0]


SMALL = [(1, 1, 1), (1, 5, 3), (33, 9, 1), (31, 7, 2), (16, 4, 5), (65, 3, 9), (129, 17, 6)]


@pytest.mark.parametrize("prec", list(TOL))
@pytest.mark.parametrize("nx,ny,nz", SMALL)
def test_small_and_ragged_cells(lblib, cuda, prec, nx, ny, nz):
    p, rho, T = _cell(prec, nx, ny, nz, nu_every=2)
    _same(prec, p, rho, T, 4)


# cells large enough to march (FP32 compute): exact tiles, one node past them, one short of them
MARCH = [(96, 96, 96), (161, 105, 90), (127, 119, 77), (64, 200, 121), (130, 99, 85), (192, 64, 128)]


@pytest.mark.parametrize("prec", ["f32", "fp16loc", "fp16dev", "bf16dev"])
@pytest.mark.parametrize("nx,ny,nz", MARCH)
@pytest.mark.parametrize("nu_every", [1, 0])     # steps that sample and plain steps are other kernels
def test_march_cells(lblib, cuda, prec, nx, ny, nz, nu_every):
    p, rho, T = _cell(prec, nx, ny, nz, nu_every=nu_every)
    _same(prec, p, rho, T, 3)


@pytest.mark.parametrize("prec", ["f64", "f32", "fp16loc"])
@pytest.mark.parametrize("forcing,psi", [(1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("nx,ny,nz", [(33, 9, 7), (97, 101, 95)])
def test_variants(lblib, cuda, prec, forcing, psi, nx, ny, nz):
    p, rho, T = _cell(prec, nx, ny, nz, forcing, psi)
    _same(prec, p, rho, T, 3)


def test_step_under_stream_capture(lblib, cuda):
    """Steps captured into a graph and replayed equal the same steps taken directly."""
    for n in (24, 96):
        p, rho, T = _cell("f32", n, n, n)
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            a, b = lb.Lattice(p, rho, T), lb.Lattice(p, rho, T)
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                a.step(2)
            # the capture ran nothing; two steps return the context to the buffers that it read
            for _ in range(3):
                graph.replay()
            b.step(6)
            fa, fb = a.populations(device=True), b.populations(device=True)
            stream.synchronize()
        assert torch.equal(fa[0], fb[0]) and torch.equal(fa[1], fb[1])
        a.close()
        b.close()
