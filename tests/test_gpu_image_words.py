"""The camera tally's 32- and 64-bit conversions: contributions below, around
and above 2^32 units give the image of a run with finer bits to within the
rounding of each contribution, and the three image modes the same words."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N, SCATTERS, FINE = 2000, 4, 48


def _image(gpu, med, bits, mode):
    e = gpu.Engine(gpu.Camera(16, 16, 8, 20.0), gpu.Geometry(40.0, 30.0, 30.0, 1.0))
    e.run(med, N, seed=5, max_scatter=SCATTERS, image_frac_bits=bits, image_mode=mode)
    e.check()
    return e.image.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("mu_a", [0.0, 0.03])
@pytest.mark.parametrize("bits", [20, 33, 38, 44])
def test_words_of_every_size(gpu, bits, mu_a):
    med = gpu.Medium(0.2, mu_a, "hg", 0.6, None)
    fine = _image(gpu, med, FINE, 2) * 2.0 ** -FINE
    imgs = [_image(gpu, med, bits, mode) for mode in (1, 2, 3)]
    assert np.array_equal(imgs[0], imgs[1]) and np.array_equal(imgs[0], imgs[2])
    # half a unit for each of the pixel's contributions, at most N x SCATTERS,
    # on both sides; a lost high word would be 2^32 units
    got = imgs[0] * 2.0 ** -bits
    assert np.max(np.abs(got - fine)) <= 0.5 * N * SCATTERS * (2.0 ** -bits + 2.0 ** -FINE)
    assert got.sum() > 0
