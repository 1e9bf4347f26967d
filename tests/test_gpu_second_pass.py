"""The gradients' second pass over a photon, which stops at its last collision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LX = 45.0
R_MAX = 5.0 * 2 ** 0.5


def _engine(gpu, nx, nz):
    return gpu.Engine(gpu.Camera(nx, nz, 128, R_MAX), gpu.Geometry(LX, 10.0, 10.0))


@pytest.mark.parametrize("kw", [dict(max_scatter=1), dict(max_scatter=2), dict(max_scatter=5), {}])
@pytest.mark.parametrize("mu_a", [0.0, 0.05])
def test_voxel_sums_match_the_homogeneous_gradient(gpu, ps_table, mu_a, kw):
    """A uniform grid walks the homogeneous medium's photons, and its voxel
    gradient sums to the gradient of the density's scale."""
    import torch
    n, rho = 200_000, np.float32(0.15)
    adj = torch.rand((32, 48), generator=torch.Generator().manual_seed(4))
    e = _engine(gpu, 48, 32)
    grid = gpu.Grid(torch.full((6, 7, 20), float(rho), device="cuda"), 1.0, 0.8, mu_a, (4, 4, 4))
    grid = grid.prepare(gpu.Geometry(LX, 10.0, 10.0))
    value, grad = e.grid_adjoint(grid, gpu.Medium(1.0, 0.0, "table", 0.0, ps_table), adj, n, seed=9, **kw)
    e.check()
    mu_s, mu_p = 0.8 * float(rho), (1.0 - 0.8) * float(rho)
    h = e.adjoint(gpu.Medium(mu_s, mu_p + mu_a, "table", 0.0, ps_table), adj, n, n_w=0, seed=9, **kw).cpu().numpy()
    e.check()
    # the bounds of the same identity without a cap, 1e6 photons
    assert float(value) == pytest.approx(h[0], rel=2e-4)
    assert float(rho) * float(grad.double().sum()) == pytest.approx(mu_s * h[1] + mu_p * h[2], rel=2e-3)


@pytest.mark.parametrize("n_bins,cell", [(64, 4), (8192, 4), (16384, 4), (8192, 1), (16384, 1)])
@pytest.mark.parametrize("n", [50, 3_000, 100_000])
def test_every_cta_size(gpu, n_bins, cell, n):
    """Few photons and large tables or many cells take other CTA sizes of the
    gradient kernel: the same identity."""
    import torch
    rho = np.float32(0.15)
    adj = torch.rand((32, 48), generator=torch.Generator().manual_seed(4))
    e = _engine(gpu, 48, 32)
    table = gpu.PhaseTable(n_bins=n_bins)
    grid = gpu.Grid(torch.full((16, 24, 32), float(rho), device="cuda"), 1.0, 0.8, 0.0, (cell, cell, cell))
    grid = grid.prepare(gpu.Geometry(LX, 10.0, 10.0))
    value, grad = e.grid_adjoint(grid, gpu.Medium(1.0, 0.0, "table", 0.0, table), adj, n, seed=9)
    e.check()
    mu_s, mu_p = 0.8 * float(rho), (1.0 - 0.8) * float(rho)
    h = e.adjoint(gpu.Medium(mu_s, mu_p, "table", 0.0, table), adj, n, n_w=0, seed=9).cpu().numpy()
    e.check()
    assert float(value) == pytest.approx(h[0], rel=2e-4)
    # few photons: the sums cancel, so against the terms' own size (the value's)
    bound = 2e-3 * abs(mu_s * h[1] + mu_p * h[2]) + 1e-3 * abs(h[0])
    assert abs(float(rho) * float(grad.double().sum()) - (mu_s * h[1] + mu_p * h[2])) <= bound


@pytest.mark.parametrize("kw", [dict(max_scatter=8), dict(max_scatter=9), dict(max_events=9), dict(max_events=10),
                                dict(max_scatter=17), {}])
@pytest.mark.parametrize("n_w,mu_a", [(5, 0.0), (256, 0.0), (64, 0.02)])
def test_angles_beyond_the_kept_ones(gpu, oracle_mod, ps_table, ps_oracle_table, n_w, mu_a, kw):
    """Photons around the eight kept angles, at an optical depth where many have
    more, against the oracle on the same photons (the bounds of the comparison
    without a cap)."""
    import torch
    n, nx, nz = 60_000, 32, 32
    mu_s = 12.0 / LX - mu_a
    adj = np.random.default_rng(8).uniform(0, 1, (nz, nx)).astype(np.float32)
    e = _engine(gpu, nx, nz)
    got = e.adjoint(gpu.Medium(mu_s, mu_a, "table", 0.0, ps_table), torch.from_numpy(adj), n, n_w=n_w, seed=5,
                    rr_threshold=0.05, **kw)
    if "max_events" not in kw:
        e.check()
    got = got.cpu().numpy()
    o = oracle_mod.adjoint(adj.astype(np.float64), n_w, mu_s=mu_s, mu_a=mu_a, table=ps_oracle_table, n_photons=n,
                           nx=nx, nz=nz, seed=5, rr_threshold=0.05, **kw)
    g = o["grad"]
    sig = np.sqrt(np.maximum(o["grad_sq"] - g ** 2 / n, 0))
    assert got[0] == pytest.approx(o["value"], rel=1e-4)
    assert np.all(np.abs(got[1:] - g) <= 0.05 * sig + 1e-4 * np.abs(g) + 1e-9)
