"""The variant for media that never change a photon's weight against the
general one. A weight threshold of 1 keeps the variant; a threshold of 2 with
certain survival takes the general walk, whose roulette then multiplies by 1:
the same photons, so the same integers. Absorption that leaves an albedo below
1 in single precision counts."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

UNIT = dict(rr_threshold=1.0, rr_survival=0.0)
GENERAL = dict(rr_threshold=2.0, rr_survival=1.0)


def _medium(gpu, phase, table, mu_a=0.0):
    if phase == "hg":
        return gpu.Medium(0.2, mu_a, "hg", 0.87)
    return gpu.Medium(0.2, mu_a, phase, 0.0, gpu.PaperTable(n_theta=500) if phase == "paper" else table)


def _state(e):
    e.check()
    return [t.cpu().numpy().copy() for t in (e.image, e.radial, e.totals)]


@pytest.mark.parametrize("phase", ["table", "hg", "paper"])
@pytest.mark.parametrize("kw", [dict(), dict(image_mode=2), dict(max_scatter=3), dict(max_events=4)])
def test_walk(gpu, ps_table, phase, kw):
    e = gpu.Engine(gpu.Camera(75, 33, 20), gpu.Geometry(45.0, 10.0, 10.0, 1.25))
    med, got = _medium(gpu, phase, ps_table), []
    for rr in (UNIT, GENERAL):
        e.run(med, 70_001, seed=3, **rr, **kw)
        if "max_events" in kw:
            with pytest.raises(Exception, match="MC_ERR_EVENTS"):
                e.check()
        got.append(_state(e))
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("phase", ["table", "hg", "paper"])
def test_grid_and_batch(gpu, ps_table, phase):
    import torch
    geo, cam = gpu.Geometry(45.0, 10.0, 10.0), gpu.Camera(75, 33, 20)
    med = _medium(gpu, phase, ps_table)
    grid = gpu.Grid(torch.rand((5, 6, 7), device="cuda") * 0.3, 1.0, 1.0, 0.0, (3, 6, 5)).prepare(geo)
    e, b, got = gpu.Engine(cam, geo), gpu.Batch(3, cam, geo), []
    for rr in (UNIT, GENERAL):
        e.run_grid(grid, med, 50_001, seed=5, **rr)
        out = _state(e)
        b.run([med] * 3, [10_001, 0, 40_000], [1, 2, 3], **rr)
        got.append(out + _state(b))
    for x, y in zip(*got):
        np.testing.assert_array_equal(x, y)


def test_absorbing_media_are_general(gpu, ps_table):
    e = gpu.Engine(gpu.Camera(16, 16, 8), gpu.Geometry(45.0, 10.0, 10.0))
    e.run(_medium(gpu, "table", ps_table, mu_a=0.05), 20_000, seed=1)
    e.check()
    r = e.result()
    assert r["totals"][3] > 100.0                        # captured weight
    b = gpu.Batch(2, gpu.Camera(16, 16, 8), gpu.Geometry(45.0, 10.0, 10.0))
    b.run([_medium(gpu, "table", ps_table), _medium(gpu, "table", ps_table, mu_a=0.05)], 20_000, seeds=1)
    b.check()
    np.testing.assert_array_equal(b.totals[1].cpu().numpy(), r["raw_totals"])
    assert int(b.totals[0, 3]) == 0


@pytest.mark.parametrize("phase,n_w", [("table", 0), ("table", 7), ("table", 200), ("hg", 0)])
def test_adjoint(gpu, ps_table, phase, n_w):
    import torch
    e = gpu.Engine(gpu.Camera(32, 20, 8), gpu.Geometry(45.0, 10.0, 10.0))
    adj = torch.linspace(0.0, 1.0, 640, device="cuda").view(20, 32)
    med = _medium(gpu, phase, ps_table)
    got = [e.adjoint(med, adj, 60_001, n_w=n_w, seed=4, **rr).cpu().numpy() for rr in (UNIT, GENERAL)]
    e.check()
    # the same terms in single precision, added in another order: compensated
    # sums, and private sums of a few terms each over the hats
    np.testing.assert_allclose(got[0], got[1], rtol=2e-6, atol=2e-6 * np.abs(got[1]).max())


def test_albedos_next_to_one(gpu, ps_table):
    """The largest single below 1 captures 2^-24 of the weight at each collision;
    an albedo that rounds to 1 captures nothing in either variant."""
    e = gpu.Engine(gpu.Camera(16, 16, 8), gpu.Geometry(45.0, 10.0, 10.0))
    n, mu = 20_000, 0.25

    def run(phase, absorbed, **rr):
        e.run(gpu.Medium(mu * (1.0 - absorbed), mu * absorbed, phase, 0.87, ps_table), n, seed=1, **rr)
        return _state(e)

    for phase in ("table", "hg"):
        totals = run(phase, 2.0 ** -24)[2]
        collisions = int(totals[7]) - n               # flights less exits: no photon is truncated
        # 2^-24 is 256 units of 2^-32; a photon's later captures are of a weight
        # that single precision holds to within 2^-24
        assert collisions > n and abs(int(totals[3]) - 256 * collisions) <= collisions
        unit, general = run(phase, 2.0 ** -26, **UNIT), run(phase, 2.0 ** -26, **GENERAL)
        assert int(unit[2][3]) == 0
        for a, b in zip(unit, general):
            np.testing.assert_array_equal(a, b)
