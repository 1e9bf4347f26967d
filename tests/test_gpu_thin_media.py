"""Gradient terms in a medium whose mean free path is far longer than the
cuvette: the score 1/mu_ext - s of a flight is then some thirty times what is
left of it in the derivative by mu_a, which may lose the score's own rounding
and no more. One photon a call, so that a call returns one term."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LX, LY = 45.0, 10.0
MFP = 1500.0


@pytest.mark.parametrize("kind,n_w", [("table", 0), ("table", 8), ("hg", 0)])
@pytest.mark.parametrize("general", [False, True])
def test_single_terms(gpu, ps_table, kind, n_w, general):
    import torch
    kw = dict(max_scatter=1)
    if general:      # roulette that multiplies by one: the variant with weights
        kw.update(rr_threshold=2.0, rr_survival=1.0)
    e = gpu.Engine(gpu.Camera(8, 8, 4), gpu.Geometry(LX, LY, 10.0))
    med = gpu.Medium(1.0 / MFP, 0.0, kind, 0.5, ps_table if kind == "table" else None)
    assert np.float32(MFP) == np.float32(1.0 / (1.0 / MFP))
    n = 4000
    t = gpu.decode_trace(e.trace(med, n, n, 1, seed=6, max_scatter=1))
    e.check()
    hit = np.nonzero(t["pix"][:, 0] >= 0)[0][:48]
    assert len(hit) == 48
    adj = torch.ones((8, 8), device="cuda")
    for p in hit:
        value, by_s, by_a = e.adjoint(med, adj, 1, n_w=n_w, seed=6, photon_offset=int(p), **kw).cpu().numpy()[:3]
        # the camera's term A and the bracket: s = x, l = ly/2 on the axis
        x, y = t["r"][p, 0, :2]
        left = -(x + LY / 2 - y)
        assert value > 0 and y == 0.0
        # 1/mu_ext - s lies in [1024, 2048): rounded to within 2^-14; its
        # difference from 1/mu_ext is exact; then one rounding of the bracket
        # and one of its product with A, each 2^-24 of itself
        assert abs(by_a / value - left) <= 2.0 ** -14 + 2.1 * 2.0 ** -24 * abs(left)
        # nothing cancels by mu_s: the score, the bracket, the product
        assert abs(by_s / value - (MFP + left)) <= 2 * 2.0 ** -14 + 1.1 * 2.0 ** -24 * MFP
    e.check()
