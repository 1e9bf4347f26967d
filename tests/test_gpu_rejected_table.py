"""A run with a table that the kernels reject stops with that error alone: the
tallies are cleared before the run ends, whatever they held, so that the check
of their signs finds no overflow and a reader no old values."""
import pytest

pytestmark = pytest.mark.gpu

N = 100_000


def _spoil(t):
    """Every tally -1 (an overflow, were it read)."""
    for a in (t.image, t.radial, t.totals):
        a.fill_(-1)


def _only_the_table(gpu, t):
    with pytest.raises(gpu._native.McError, match="MC_ERR_TABLE"):
        t.check()
    for a in (t.image, t.radial, t.totals):
        assert not bool(a.any())


def _rejected(gpu, base):
    import torch
    w = torch.ones(16, device="cuda")
    w[3] = 0.0
    return gpu.Medium(0.2, 0.0, "table", 0.0, gpu.WeightedTable(base, w))


@pytest.mark.parametrize("side", [64, 1024])
@pytest.mark.parametrize("n", [1, N])
def test_walk_and_grid(gpu, ps_table, side, n):
    import torch
    geo = gpu.Geometry(45.0, 10.0, 10.0)
    e, med = gpu.Engine(gpu.Camera(side, side, 32), geo), _rejected(gpu, ps_table)
    grid = gpu.Grid(torch.full((4, 4, 8), 0.2, device="cuda"), 1.0, 1.0, 0.0, (8, 4, 4)).prepare(geo)
    for run in (lambda: e.run(med, n, seed=1), lambda: e.run_grid(grid, med, n, seed=1)):
        _spoil(e)
        run()
        _only_the_table(gpu, e)
        assert e.last_error == gpu._native.EFLAG_TABLE


@pytest.mark.parametrize("side", [64, 1024])
def test_batch(gpu, ps_table, side):
    b = gpu.Batch(3, gpu.Camera(side, side, 32), gpu.Geometry(45.0, 10.0, 10.0))
    _spoil(b)
    b.run([_rejected(gpu, ps_table)] * 3, N, seeds=1)
    _only_the_table(gpu, b)
