"""How a batch shares its CTAs out among the media: budgets from nothing over
a warp's remainders to far more than one CTA's share, one medium or many per
CTA, fresh and added-to tallies; every medium's integers equal a plain run's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = {
    "tiny": [0, 1, 31, 32, 33, 127, 128, 129] * 8,
    "one-large": [1] * 20 + [2_000_000] + [0] * 20 + [500],
    "one-medium": [5_000],
    "nothing": [0, 0, 0],
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("kw", [dict(), dict(block_size=32, blocks_per_sm=1), dict(item_photons=4096)])
def test_every_medium_is_run_once(gpu, ps_table, name, kw):
    nph = CASES[name]
    cam, geo = gpu.Camera(37, 21, 9), gpu.Geometry(45.0, 10.0, 10.0)
    media = [gpu.Medium((0.5 + (i % 7) * 3.0) / 45.0, 0.0, "table", 0.0, ps_table) for i in range(len(nph))]
    b = gpu.Batch(len(nph), cam, geo)
    b.run(media, nph, list(range(len(nph))), image_frac_bits=24, **kw)
    b.run(media, nph, list(range(len(nph))), offsets=7, image_frac_bits=24, accumulate=True, **kw)
    b.check()
    e = gpu.Engine(cam, geo)
    for i, med in enumerate(media):
        if i % 8 > 4 and name == "tiny" and i > 16:
            continue
        e.run(med, nph[i], seed=i, image_frac_bits=24)
        e.run(med, nph[i], seed=i, photon_offset=7, image_frac_bits=24, accumulate=True)
        e.check()
        for got, want in ((b.image, e.image), (b.radial, e.radial), (b.totals, e.totals)):
            np.testing.assert_array_equal(got[i].cpu().numpy(), want.cpu().numpy(), err_msg="medium %d" % i)
