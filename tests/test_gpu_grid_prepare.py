"""The prepared grid against numpy in double precision, bit for bit: voxel
coefficients, the optical depth above each voxel (double sums, rounded once)
and the majorants, for voxel heights whose products are exact in double
precision and ones that round, cells that end inside the grid, columns that do
not fill a warp, and densities with zeros, subnormal and huge values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,block,ly", [((1, 1, 1), (1, 1, 1), 10.0), ((3, 5, 7), (2, 3, 2), 10.0),
                                            ((5, 64, 33), (8, 16, 16), 10.0), ((9, 67, 101), (101, 67, 9), 7.3),
                                            ((2, 9, 40), (3, 1, 1), 1.0 / 3.0), ((4, 256, 64), (32, 256, 4), 10.0)])
@pytest.mark.parametrize("values", ["plain", "extreme"])
def test_prepared_grid_is_exact(gpu, shape, block, ly, values):
    import torch
    gz, gy, gx = shape
    rng = np.random.default_rng(gx * 1000 + gy)
    d = np.exp(rng.standard_normal(shape)).astype(np.float32)
    if values == "extreme":
        pick = rng.integers(0, 5, shape)
        d = np.where(pick == 0, 0.0, np.where(pick == 1, 1e-42, np.where(pick == 2, 1e-37, np.where(pick == 3, 1e30, d)))
                     ).astype(np.float32)
    k_ext, mu_a = 0.7, 0.0 if values == "extreme" else 0.013
    grid = gpu.Grid(torch.from_numpy(d).cuda(), k_ext, k_ext, mu_a, block).prepare(gpu.Geometry(45.0, ly, 10.0))
    torch.cuda.synchronize()
    raw = grid.work.cpu().numpy()
    cells = raw[:8 * gx * gy * gz].view(np.float32).reshape(gz, gy, gx, 2)
    # fmaf(k_ext, n, mu_a): exact in double for 24-bit factors, then one rounding
    mu = (np.float64(np.float32(k_ext)) * d.astype(np.float64) + np.float64(np.float32(mu_a))).astype(np.float32)
    np.testing.assert_array_equal(cells[..., 0], mu)
    vy, od = ly / gy, np.zeros((gz, gx))
    for iy in range(gy - 1, -1, -1):
        with np.errstate(over="ignore"):
            np.testing.assert_array_equal(cells[:, iy, :, 1], od.astype(np.float32))
        od = od + mu[:, iy, :].astype(np.float64) * vy
    bx, by, bz = block
    mx, my, mz = -(-gx // bx), -(-gy // by), -(-gz // bz)
    off = (8 * gx * gy * gz + 15) // 16 * 16
    maj = raw[off:off + 4 * mx * my * mz].view(np.float32).reshape(mz, my, mx)
    for cz in range(mz):
        for cy in range(my):
            for cx in range(mx):
                part = mu[cz * bz:(cz + 1) * bz, cy * by:(cy + 1) * by, cx * bx:(cx + 1) * bx]
                assert maj[cz, cy, cx] == part.max()
