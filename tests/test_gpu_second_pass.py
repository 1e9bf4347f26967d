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
