"""Image metrics at the sizes where the pixel split can go wrong: runs of 8
pixels that end inside a row, image or CTA; ring sums in shared memory (up to
512 rings) or straight to L2; images at any 8-byte address; values over the
whole range that doubles hold exactly, negative ones included."""
import numpy as np
import pytest

from oracle import metrics as OM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz,nx,n_r", [(1, 1, 4096), (1, 9, 3), (9, 1, 2), (3, 5, 512), (17, 129, 513), (64, 64, 4096),
                                       (600, 500, 31), (2, 4099, 100)])
@pytest.mark.parametrize("with_b", [True, False])
def test_image_metrics_sizes(gpu, nz, nx, n_r, with_b):
    import torch
    rng = np.random.default_rng(nz * 10007 + nx * 31 + n_r)
    ims = [rng.integers(-(1 << 52), 1 << 52, size=(nz, nx), dtype=np.int64) for _ in range(3)]
    ims[1] = ims[0] // 3 + ims[1] // 5
    dev = []
    for a in ims:       # one element past a 256-byte boundary: only 8-byte aligned
        buf = torch.empty(nz * nx + 1, dtype=torch.int64, device="cuda")
        buf[1:] = torch.from_numpy(a.reshape(-1)).cuda()
        dev.append(buf[1:].view(nz, nx))
    got = gpu.image_metrics(dev[0], dev[1], dev[2] if with_b else None, n_r=n_r)
    want = OM.compare(ims[0], ims[1], ims[2] if with_b else None, n_r=n_r)
    # sums of at most 3e5 doubles in another order: below 3e5 x 2^-53 relative
    # to sums of the same sign, 1e-13 absolute for centred ones (values <= 1)
    np.testing.assert_allclose(got, want, rtol=1e-10, atol=1e-12)


def test_image_metrics_identical_images_are_zero_apart(gpu):
    import torch
    a = torch.randint(0, 1 << 45, (77, 130), dtype=torch.int64, device="cuda")
    got = gpu.image_metrics(a, a.clone(), a.clone(), n_r=20)
    assert got[0] == 0.0 and got[6] == 0.0 and np.all(got[2:5] == 0.0)
    assert abs(got[1] - 1.0) < 1e-14 and got[12] == 0.0
