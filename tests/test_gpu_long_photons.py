"""Photons around the flight count from which the walk looks at its counters
(2^16): one more flight allowed is one more flight of exactly the photons that
the shorter limit ended."""
import pytest

pytestmark = pytest.mark.gpu

N, EDGE = 4000, 1 << 16


@pytest.mark.parametrize("kind", ["unit", "roulette", "grid", "batch"])
def test_one_more_flight(gpu, kind):
    import torch
    geo, cam = gpu.Geometry(45.0, 10.0, 10.0), gpu.Camera(8, 8, 4)
    # isotropic and far thicker than 1 / 2^8 mm: some photons stay for 2^16 flights
    med = gpu.Medium(3000.0, 0.0, "hg", 0.0, None)
    e = gpu.Batch(2, cam, geo) if kind == "batch" else gpu.Engine(cam, geo)
    grid = gpu.Grid(torch.full((2, 2, 4), 3000.0, device="cuda"), 1.0, 1.0, 0.0, (4, 2, 2)).prepare(geo)
    kw = dict(rr_threshold=2.0, rr_survival=1.0) if kind == "roulette" else {}

    def run(limit):
        if kind == "grid":
            e.run_grid(grid, med, N, seed=3, max_events=limit)
        elif kind == "batch":
            e.run([med] * 2, [N, 0], seeds=3, max_events=limit)
        else:
            e.run(med, N, seed=3, max_events=limit, **kw)
        with pytest.raises(Exception, match="MC_ERR_EVENTS"):
            e.check()
        t = (e.totals[0] if kind == "batch" else e.totals).cpu().numpy()
        assert int(t[0]) + int(t[1]) + int(t[2]) + int(t[5]) == N << 32
        return int(t[5]) >> 32, int(t[7])

    runs = [run(EDGE + d) for d in (-2, -1, 0, 1, 2)]
    assert 0 < runs[-1][0] < N
    for (cut, steps), (_, more) in zip(runs, runs[1:]):
        assert more - steps == cut
