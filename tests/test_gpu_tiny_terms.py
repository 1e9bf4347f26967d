"""Gradient terms at the bottom of the single-precision range: those of a density
gradient add nothing beyond their own size, and camera transmittances below
2^-126 still count in the gradients of the coefficients."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nulls", [None, 1.5])
@pytest.mark.parametrize("power", [-100, -130, -145])
def test_terms_below_the_normal_range(gpu, ps_table, nulls, power):
    import torch
    geo = gpu.Geometry(45.0, 10.0, 10.0)
    e = gpu.Engine(gpu.Camera(16, 16, 8), geo)
    grid = gpu.Grid(torch.full((12, 40, 16), 0.2, device="cuda"), 1.0, 1.0, 0.0, (4, 8, 4)).prepare(geo)
    med = gpu.Medium(1.0, 0.0, "table", 0.0, ps_table)

    def gradient(adj):
        _, grad = e.grid_adjoint(grid, med, torch.full((16, 16), adj), 20_000, seed=2, nulls=nulls)
        e.check()
        return grad.double().cpu().numpy()

    one, small = gradient(1.0), gradient(2.0 ** power)
    size = np.abs(one).sum() * 2.0 ** power
    if power == -100:
        # the same photons; a term comes from a product of four numbers at most,
        # of which 2^-100 takes none out of the normal range but the smallest
        np.testing.assert_allclose(small * 2.0 ** 100, one, rtol=1e-4, atol=1e-6 * np.abs(one).max())
    # terms that are too small are dropped or rounded to multiples of 2^-149:
    # an entry is then off by its terms' own size at most, which cancellation
    # may leave 2^10 times the entries', plus half a unit
    assert np.abs(small).sum() <= 2.0 ** 10 * size + one.size * 2.0 ** -149


@pytest.mark.parametrize("n_w", [0, 8])
def test_transmittance_below_the_normal_range_counts(gpu, n_w, ps_table):
    """One scatter on the axis of a medium 92 free paths below the camera face:
    exp(-92) is 1.1e-40, and adjoint pixels of 1e38 bring the terms back."""
    import torch
    ly, mu = 10.0, 18.4
    e = gpu.Engine(gpu.Camera(4, 4, 4), gpu.Geometry(45.0, ly, ly))
    med = gpu.Medium(mu, 0.0, "table", 0.0, ps_table)
    n = 2000
    v = e.adjoint(med, torch.full((4, 4), 1e38), n, n_w=n_w, seed=3, max_scatter=1).cpu().numpy()[0]
    e.check()
    # every photon collides; the density for the camera direction at the beam
    j = int(np.searchsorted(ps_table.icdf64, 0.0, side="right")) - 1
    psr, t = float(ps_table.pdf64[j]) / (2 * math.pi), math.exp(-mu * ly / 2)
    want = n * 1e38 * psr * t
    # the transmittance and its product with the density are rounded to multiples
    # of 2^-149; its exponent of 133 binary digits to 2^-17 each in two steps
    rel = 0.5 * 2.0 ** -149 / t + 0.5 * 2.0 ** -149 / (psr * t) + 2 * 133 * 2.0 ** -24
    assert rel < 2e-3
    assert v == pytest.approx(want, rel=rel)
