"""Flights cut into pieces at voxel planes: the pieces of a flight add up to its
length whatever the voxels, so sum(n dL/dn) over a uniform medium does not
depend on the grid (the same photons: the majorant is the medium's own
coefficient everywhere). Grids with one voxel along an axis, fewer and more
than the 32 voxels of the box around the beam, odd counts, and a disc beam."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 2), (1, 64, 1), (33, 1, 70), (2, 3, 300), (31, 32, 33), (64, 50, 17), (100, 7, 5)])
@pytest.mark.parametrize("beam", [0.0, 2.5])
def test_pieces_add_up(gpu, ps_table, shape, beam):
    import torch
    geo, cam = gpu.Geometry(45.0, 10.0, 12.0, beam), gpu.Camera(16, 12, 8)
    e = gpu.Engine(cam, geo)
    med = gpu.Medium(1.0, 0.0, "table", 0.0, ps_table)
    adj = torch.linspace(0.5, 1.5, 12 * 16, device="cuda").view(12, 16)
    got = []
    for s in ((1, 1, 1), shape):
        gz, gy, gx = s
        grid = gpu.Grid(torch.full(s, 0.2, device="cuda"), 1.0, 0.9, 0.0, (gx, gy, gz)).prepare(geo)
        value, grad = e.grid_adjoint(grid, med, adj, 30_000, seed=2)
        e.check()
        assert bool(torch.isfinite(grad).all())
        got.append((float(value), float((0.2 * grad.double()).sum()), float((0.2 * grad.double()).abs().sum())))
    assert got[1][0] == pytest.approx(got[0][0], rel=1e-5)
    # single-precision lengths of millions of pieces: 2^-24 of each piece's terms, against the sum of magnitudes
    # (positions near voxel planes and camera columns round differently on each grid)
    assert abs(got[1][1] - got[0][1]) <= 2e-5 * (abs(got[0][1]) + got[1][2])
