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


@pytest.mark.parametrize("mu_a", [0.0, 0.03])
@pytest.mark.parametrize("bits", [20, 32, 44, 48])
def test_every_unit_counts(gpu, bits, mu_a):
    """The image is the sum of the traced camera terms, each rounded to units of
    2^-bits, to the last unit: on both sides of the 32-bit conversion."""
    med = gpu.Medium(0.2, mu_a, "hg", 0.6, None)
    e = gpu.Engine(gpu.Camera(16, 16, 8, 20.0), gpu.Geometry(40.0, 30.0, 30.0, 1.0))
    t = gpu.decode_trace(e.trace(med, N, N, SCATTERS + 1, seed=5, max_scatter=SCATTERS))
    e.check()
    hit = t["pix"] >= 0
    terms = np.rint(t["nee"][hit] * 2.0 ** bits).astype(np.int64)     # exact products, halves to even
    want = np.zeros(256, np.int64)
    np.add.at(want, t["pix"][hit], terms)
    if bits == 44:
        assert terms.min() < 1 << 32 < terms.max()
    for mode in (1, 2, 3):
        e.run(med, N, seed=5, max_scatter=SCATTERS, image_frac_bits=bits, image_mode=mode)
        e.check()
        np.testing.assert_array_equal(e.image.cpu().numpy().reshape(-1), want)
