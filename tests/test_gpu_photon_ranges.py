"""How a launch hands its photon range out to warps (first chunks by warp
number, later ones from a counter, chunk sizes that fall toward the end): at
the edges of a warp, of the first chunks and of the chip's lanes every photon
runs exactly once, whatever the launch shape."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LANES = 152 * 1024


@pytest.mark.parametrize("n", [1, 31, 33, 152 * 32 - 1, 152 * 32 + 1, 152 * 256 + 1, LANES - 1, LANES + 1, 2 * LANES + 1,
                               6 * LANES + 17])
def test_walk_range(gpu, ps_table, n):
    med = gpu.Medium(2.0 / 45.0, 0.0, "table", 0.0, ps_table)
    e = gpu.Engine(gpu.Camera(40, 24, 8), gpu.Geometry(45.0, 10.0, 10.0))
    got = []
    for kw in (dict(), dict(block_size=32, blocks_per_sm=1), dict(block_size=96)):
        e.run(med, n, seed=4, photon_offset=(1 << 33) - 5, **kw)
        e.check()
        got.append((e.image.cpu().numpy(), e.totals.cpu().numpy(), e.radial.cpu().numpy()))
    t = got[0][1]
    assert int(t[0]) + int(t[1]) + int(t[2]) == n << 32     # no absorption: every photon leaves, once
    for other in got[1:]:
        for a, b in zip(got[0], other):
            np.testing.assert_array_equal(a, b)
    cut = n // 3                                            # the same photons in two calls
    e.run(med, cut, seed=4, photon_offset=(1 << 33) - 5, image_frac_bits=e.image_frac_bits)
    e.run(med, n - cut, seed=4, photon_offset=(1 << 33) - 5 + cut, accumulate=True)
    e.check()
    np.testing.assert_array_equal(e.image.cpu().numpy(), got[0][0])
    np.testing.assert_array_equal(e.totals.cpu().numpy(), t)


@pytest.mark.parametrize("n", [1, 33, 152 * 32 + 1, LANES + 1])
def test_grid_and_adjoint_ranges(gpu, ps_table, n):
    import torch
    cam, geo = gpu.Camera(16, 16, 8), gpu.Geometry(45.0, 10.0, 10.0)
    e = gpu.Engine(cam, geo)
    med = gpu.Medium(0.1, 0.0, "table", 0.0, ps_table)
    adj = torch.ones((16, 16), device="cuda")
    e.run(med, n, seed=9, image_frac_bits=32)
    e.check()
    want = float(e.image.double().sum()) * 2.0 ** -32
    g = e.adjoint(med, adj, n, n_w=0, seed=9)
    gw = e.adjoint(med, adj, n, n_w=16, seed=9)
    # the camera terms' sum: each image pixel rounds a term to 2^-32, the
    # gradient's sums are compensated single precision
    assert abs(float(g[0]) - want) <= 1e-5 * abs(want) + n * 2.0 ** -32
    assert abs(float(gw[0]) - want) <= 1e-5 * abs(want) + n * 2.0 ** -32
    grid = gpu.Grid(torch.full((4, 4, 8), 0.1, device="cuda"), 1.0, 1.0, 0.0, (8, 4, 4)).prepare(geo)
    e.run_grid(grid, med, n, seed=9, image_frac_bits=32)
    e.check()
    assert int(e.totals[:3].sum()) == n << 32
    want = float(e.image.double().sum()) * 2.0 ** -32
    for nulls in (None, 1.25):
        value, _ = e.grid_adjoint(grid, med, adj, n, seed=9, nulls=nulls)
        if nulls is None:       # scaled majorants draw other paths
            assert abs(float(value) - want) <= 1e-5 * abs(want) + n * 20 * 2.0 ** -32
        cut = n // 3            # the same photons in two calls; their terms are
        parts = [float(e.grid_adjoint(grid, med, adj, m, seed=9, nulls=nulls, photon_offset=o)[0])
                 for m, o in ((cut, 0), (n - cut, cut))]       # summed in double
        assert abs(float(value) - sum(parts)) <= n * 2.0 ** -53 * abs(float(value))
    e.check()
