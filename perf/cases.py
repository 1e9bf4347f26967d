"""The work that a program using this framework has it do, as cases that can be timed and compared.

Every case goes through the public entry points (Engine, Batch, Grid, run_host, camera_image,
image_metrics). listed() holds twelve of them, from a call of 20 000 photons to the 1e8-photon headline
walk; draw() gives more over the same ranges. The photons' seed, the media, the density fields, the
adjoint images and the phase weights are made from the seed; the phase tables are the plan that such a
program builds once and keeps.

Tallies of the walks are 64-bit fixed-point integers that do not depend on launch shape or order, so
they are compared exactly. The gradients and the metrics are floating point; exact() evaluates them in
64 bits with torch and numpy alone: Lorenz-Mie series, inverse-CDF table, Philox numbers, the walk and
its likelihood-ratio gradients.
"""
import functools
import math

import numpy as np
import torch

import paper_2507_23189_gb300 as mc

N_MEDIUM, N_PARTICLE, WAVELENGTH_NM = 1.33, 1.59, 532.0
RR_THRESHOLD, RR_SURVIVAL = 1e-4, 0.1
K_EXT = 4.2e-5                    # mm^2, cross section of a 5 um polystyrene sphere in water
HG_G = 0.87                       # close to the Mie g of those spheres
R_MAX = 5.0 * 2 ** 0.5


def _walk(name, **kw):
    c = dict(kind="walk", phase="mie", diameter_um=5.0, n_bins=4096, tau=5.0, albedo=1.0, n=1_000_000, nx=128,
             nz=128, n_radial=128, lx=45.0, ly=10.0, lz=10.0, beam_radius=0.0, cut=False)
    return dict(c, name=name, **kw)


def listed():
    return [
        # the smallest call: a preview, or one of many short calls of an interactive program
        _walk("call-20k", tau=1.0, n=20_000, nx=64, nz=64),
        # the small optical-depth-1 workload from host buffers to host buffers, as a C or numpy caller has it
        _walk("host-1e6", kind="host", tau=1.0, n=1_000_000, nx=64, nz=64),
        # the headline: one production image at optical depth 5
        _walk("walk-tau5-1e8", n=100_000_000, nx=256, nz=256),
        # the analytic phase function in a thick, absorbing suspension (weights, roulette), ragged sizes
        _walk("walk-hg-absorbing", phase="hg", tau=20.0, albedo=0.95, n=3_000_017, nx=301, nz=97, n_radial=77),
        # the paper's own set-up: 3000-angle table searched by bisection, 2.5 mm beam, plain cut
        _walk("walk-paper-setup", phase="paper", tau=8.0, n=10_000_000, nx=60, nz=90, lx=30.0, ly=10.0, lz=45.0,
              beam_radius=1.25, cut=True),
        # dilution series: 8 particle sizes x 8 optical depths in one launch, short budgets
        dict(name="batch-64", kind="batch", media=64, n=200_000, nx=128, nz=128),
        # gradient with respect to the two coefficients: one step of a (mu_s, mu_a) fit
        _walk("adjoint-mu", kind="adjoint", n=10_000_000, n_w=0),
        # a training step through autograd: forward image and gradient of mu_s, mu_a and 64 phase weights
        _walk("fit-step-64w", kind="fit", albedo=0.98, n=1_000_000, n_w=64),
        # a heterogeneous medium (Gaussian plume of peak optical depth 30) that was prepared once, imaged
        dict(name="plume-walk", kind="grid-walk", gx=256, gy=256, gz=256, bx=32, by=256, bz=256, tau=30.0, albedo=1.0,
             mu_a=0.0, n=20_000_000, nx=512, nz=512),
        # one step of a density reconstruction on that plume: new densities prepared, gradient of every voxel
        dict(name="plume-gradient", kind="grid-grad", gx=256, gy=256, gz=256, bx=32, by=256, bz=256, tau=30.0,
             albedo=1.0, mu_a=0.0, n=2_000_000, nx=512, nz=512, nulls=0.0),
        # the same step with null-collision scores on a small ragged grid with absorption, image included
        dict(name="grid-step-nulls", kind="grid-step", gx=101, gy=67, gz=83, bx=8, by=16, bz=16, tau=10.0, albedo=0.95,
             mu_a=0.005, n=500_000, nx=96, nz=120, nulls=1.25),
        # Tables 3 and 4: two models' images against a reference, normalised, RMSE, r, radial zones
        dict(name="metrics-512", kind="metrics", nx=512, nz=512, n_r=32),
    ]


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["walk", "walk", "walk", "host", "batch", "adjoint", "fit", "grid-walk", "grid-grad", "grid-step",
                       "metrics"])
    if kind == "metrics":
        return dict(kind=kind, nx=logint(48, 1024), nz=logint(48, 1024), n_r=logint(8, 128))
    if kind == "batch":
        return dict(kind=kind, media=rng.randint(8, 64), n=logint(20_000, 1_000_000), nx=logint(32, 200),
                    nz=logint(32, 200))
    if kind.startswith("grid"):
        c = dict(kind=kind, gx=logint(24, 256), gy=logint(24, 256), gz=logint(24, 256), tau=round(rng.uniform(1.0, 30.0), 2),
                 albedo=rng.choice([1.0, round(rng.uniform(0.9, 1.0), 3)]), mu_a=rng.choice([0.0, 0.005]),
                 n=logint(50_000, 2_000_000), nx=logint(32, 512), nz=logint(32, 512))
        if rng.random() < 0.5:      # slabs along the beam, or blocks
            c.update(bx=max(4, c["gx"] // 8), by=c["gy"], bz=c["gz"])
        else:
            c.update(bx=16, by=32, bz=32)
        if kind != "grid-walk":
            c["nulls"] = rng.choice([0.0, 1.25])
        return c
    c = _walk("", kind=kind, tau=round(rng.uniform(0.5, 20.0), 2), nx=logint(32, 400), nz=logint(32, 400),
              n_radial=logint(16, 256), albedo=rng.choice([1.0, 1.0, round(rng.uniform(0.9, 0.999), 4)]),
              beam_radius=rng.choice([0.0, 1.25]))
    del c["name"]
    if kind in ("walk", "host"):
        c.update(phase=rng.choice(["mie", "mie", "hg", "paper"]), cut=rng.random() < 0.2, n_bins=rng.choice([1024, 4096]),
                 n=logint(10_000, 40_000_000 if kind == "walk" else 4_000_000))
        if rng.random() < 0.2:      # the paper's cuvette
            c.update(lx=30.0, ly=10.0, lz=45.0)
    elif kind == "adjoint":
        c.update(phase=rng.choice(["mie", "hg"]), n=logint(100_000, 10_000_000))
        c["n_w"] = rng.choice([0, 64, logint(4, 128)]) if c["phase"] == "mie" else 0
    else:
        c.update(n=logint(100_000, 2_000_000), n_w=rng.choice([0, 16, 64]))
    return c


# ------------------------------------------------------------------ plans


@functools.lru_cache(maxsize=64)
def _table(diameter_um, n_bins):
    return mc.PhaseTable(diameter_um, N_PARTICLE, N_MEDIUM, WAVELENGTH_NM, n_bins)


@functools.lru_cache(maxsize=1)
def _paper_table():
    return mc.PaperTable(5.0, N_PARTICLE, N_MEDIUM, WAVELENGTH_NM)


def _sizes(media):
    return [(1.0 * 10.0 ** ((i % 8) / 7.0), 1.0 + 19.0 * (i // 8) / max(1, (media - 1) // 8)) for i in range(media)]


def _coefficients(case, seed):
    """mu_s, mu_a of the medium that a seed stands for: within 5 % of the case's optical depth."""
    f = 1.0 + 0.05 * (2.0 * np.random.RandomState(seed % (1 << 31)).rand() - 1.0)
    mu = case["tau"] * f / case.get("lx", 45.0)
    return mu * case["albedo"], mu * (1.0 - case["albedo"])


def _medium(case, seed):
    mu_s, mu_a = _coefficients(case, seed)
    if case["phase"] == "hg":
        return mc.Medium(mu_s, mu_a, "hg", HG_G)
    if case["phase"] == "paper":
        return mc.Medium(mu_s, mu_a, "paper", 0.0, _paper_table())
    return mc.Medium(mu_s, mu_a, "table", 0.0, _table(case["diameter_um"], case["n_bins"]))


def _random(seed, shape, lo, hi):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return lo + (hi - lo) * torch.rand(shape, generator=g, device="cuda", dtype=torch.float32)


def _density(case, seed):
    """A Gaussian plume on the beam axis (sigma 5 mm) with a few per cent of voxel noise, scaled to the case's
    optical depth along the beam; the seed moves it along the beam and sets the noise."""
    gx, gy, gz = case["gx"], case["gy"], case["gz"]
    x0 = 22.5 + 3.0 * (2.0 * np.random.RandomState(seed % (1 << 31)).rand() - 1.0)

    def axis(n, length, centre):
        p = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * (length / n) - centre
        return torch.exp(-0.5 * (p / 5.0) ** 2)

    d = (axis(gz, 10.0, 5.0)[:, None, None] * axis(gy, 10.0, 5.0)[None, :, None] * axis(gx, 45.0, x0)[None, None, :])
    peak = case["tau"] / (K_EXT * float(axis(gx, 45.0, x0).sum()) * 45.0 / gx)
    return (peak * d).float() * _random(seed, (gz, gy, gx), 0.95, 1.05)


def _adjoint_image(case, seed):
    return _random(seed + 1, (case["nz"], case["nx"]), 0.0, 1.0)


def _weights(case, seed):
    return _random(seed + 2, (case["n_w"],), 0.5, 1.5).double()


def _geometry(case):
    return mc.Geometry(case.get("lx", 45.0), case.get("ly", 10.0), case.get("lz", 10.0), case.get("beam_radius", 0.0))


def _camera(case):
    return mc.Camera(case["nx"], case["nz"], case.get("n_radial", 128), R_MAX)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, seed=seed)
    if kind == "metrics":
        # side images as the walk leaves them: int64 fixed point, bright along the beam, noisy
        z = torch.arange(case["nz"], device="cuda", dtype=torch.float64)[:, None] / case["nz"] - 0.5
        x = torch.arange(case["nx"], device="cuda", dtype=torch.float64)[None, :] / case["nx"]
        s["images"] = [((2.0 ** 32) * torch.exp(-(3.0 + k) * x - torch.abs(z) * 20.0)
                        * _random(seed + k, (case["nz"], case["nx"]), 0.5, 1.5).double()).to(torch.int64) for k in range(3)]
        return s
    cam, geo = _camera(case), _geometry(case)
    if kind == "batch":
        rnd = np.random.RandomState(seed % (1 << 31))
        sizes = _sizes(case["media"])
        s["media"] = [mc.Medium(t * (0.95 + 0.1 * rnd.rand()) / 45.0, 0.0, "table", 0.0, _table(d, 4096)) for d, t in sizes]
        for m in s["media"]:
            m.table.device_blob("cuda")
        s["batch"] = mc.Batch(case["media"], cam, geo, "cuda")
        return s
    if kind.startswith("grid"):
        s["density"] = _density(case, seed)
        s["grid"] = mc.Grid(s["density"], K_EXT, K_EXT * case["albedo"], case["mu_a"], (case["bx"], case["by"], case["bz"]))
        s["phase"] = mc.Medium(1.0, 0.0, "table", 0.0, _table(5.0, 4096))
        s["phase"].table.device_blob("cuda")
        s["geometry"] = geo
        s["engine"] = mc.Engine(cam, geo, "cuda")
        if kind == "grid-walk":
            s["grid"].prepare(geo)
        else:
            s["adj"] = _adjoint_image(case, seed)
        return s
    s["medium"] = _medium(case, seed)
    if case["phase"] != "hg":
        s["medium"].table.device_blob("cuda")
    s["kw"] = dict(rr_threshold=1e-3, rr_survival=0.0) if case["cut"] else dict(rr_threshold=RR_THRESHOLD,
                                                                               rr_survival=RR_SURVIVAL)
    if kind == "host":
        s["camera"], s["geometry"] = cam, geo
        s["work"] = torch.empty(mc.host_workspace_bytes(s["medium"], cam), dtype=torch.uint8, device="cuda")
        pinned = [torch.zeros(n, dtype=torch.int64).pin_memory() for n in (cam.nz * cam.nx, cam.n_radial, 8)]
        s["image"], s["radial"], s["totals"] = pinned[0].numpy().reshape(cam.nz, cam.nx), pinned[1].numpy(), pinned[2].numpy()
        s["pinned"] = pinned
        return s
    s["engine"] = mc.Engine(cam, geo, "cuda")
    if kind in ("adjoint", "fit"):
        s["adj"] = _adjoint_image(case, seed)
        s["w"] = _weights(case, seed) if case["n_w"] else None
    return s


def run(s):
    case, kind, n = s["case"], s["case"]["kind"], s["case"].get("n")
    if kind == "metrics":
        return mc.image_metrics(*s["images"], n_r=case["n_r"])
    if kind == "walk":
        e = s["engine"]
        e.run(s["medium"], n, seed=s["seed"], **s["kw"])
        return [e.image, e.radial, e.totals]
    if kind == "host":
        return list(mc.run_host(s["medium"], s["geometry"], s["camera"], n, s["work"], seed=s["seed"], image=s["image"],
                                radial=s["radial"], totals=s["totals"], **s["kw"]))
    if kind == "batch":
        b = s["batch"]
        b.run(s["media"], n, seeds=s["seed"])
        return [b.image, b.radial, b.totals]
    if kind == "adjoint":
        return s["engine"].adjoint(s["medium"], s["adj"], n, n_w=case["n_w"], seed=s["seed"], phase_w=s["w"], **s["kw"])
    if kind == "fit":
        mu_s = torch.tensor(s["medium"].mu_s, dtype=torch.float64, requires_grad=True)
        mu_a = torch.tensor(s["medium"].mu_a, dtype=torch.float64, requires_grad=True)
        w = s["w"].detach().clone().requires_grad_(True) if s["w"] is not None else None
        img = mc.camera_image(s["engine"], s["medium"].table, mu_s, mu_a, w, n_photons=n, seed=s["seed"],
                              grad_seed=s["seed"] + 1, **s["kw"])
        img.backward(s["adj"].double())
        return [img.detach(), mu_s.grad, mu_a.grad] + ([w.grad] if w is not None else [])
    e, grid = s["engine"], s["grid"]
    kw = dict(rr_threshold=RR_THRESHOLD, rr_survival=RR_SURVIVAL)
    if kind == "grid-walk":
        e.run_grid(grid, s["phase"], n, seed=s["seed"], **kw)
        return [e.image, e.radial, e.totals]
    grid.prepare(s["geometry"])
    out = []
    if kind == "grid-step":
        e.run_grid(grid, s["phase"], n, seed=s["seed"], **kw)
        out = [e.image, e.radial, e.totals]
    value, grad = e.grid_adjoint(grid, s["phase"], s["adj"], n, seed=s["seed"], nulls=case["nulls"] or None, **kw)
    return out + [value, grad]


# ------------------------------------------------------------------ work and tolerance


def _steps(tau):
    """Sampled flights per photon at optical depth tau in this cuvette (measured with the walk)."""
    return float(np.interp(tau, [0.0, 0.5, 1, 2, 5, 10, 20, 30], [1.0, 1.5, 1.9, 2.65, 4.3, 6.1, 8.8, 11.0]))


# arithmetic of one photon-step, each operation counted once: Philox 80, logarithm and flight 12, walls 8,
# camera term and pixel 20, table or closed-form angle 10, rotation 50, tallies 20
STEP_OPS = 200.0


def work(case):
    kind = case["kind"]
    if kind == "metrics":
        px = case["nx"] * case["nz"]
        return dict(bytes=3 * 8.0 * px + 8.0 * (13 + 3 * case["n_r"]), flops=3.0 * px * 30)
    img = 8.0 * case["nx"] * case["nz"]
    if kind == "batch":
        return dict(bytes=case["media"] * (img + 41056.0),
                    flops=STEP_OPS * case["n"] * sum(_steps(t) for _, t in _sizes(case["media"])))
    if kind.startswith("grid"):
        vox = float(case["gx"] * case["gy"] * case["gz"])
        walks = {"grid-walk": 1.0, "grid-grad": 1.0, "grid-step": 2.0}[kind]
        # the densities read, one 8-byte voxel record gathered per collision; a gradient writes every voxel and
        # reads and writes one sum per voxel
        coll = case["n"] * _steps(case["tau"])
        by = 8.0 * min(vox, coll) + (img if kind != "grid-grad" else img / 2)
        if kind != "grid-walk":
            by += 4.0 * vox + 4.0 * vox
        return dict(bytes=by, flops=STEP_OPS * walks * coll)
    steps = case["n"] * _steps(case["tau"])
    by = img + 8.0 * case["n_radial"] + (0.0 if case["phase"] == "hg" else 10.0 * case["n_bins"])
    if kind == "adjoint":
        by = img / 2 + 8.0 * (3 + case["n_w"]) + 10.0 * case["n_bins"]
    return dict(bytes=by, flops=STEP_OPS * steps * (2.0 if kind == "fit" else 1.0))


def tolerance(case):
    kind = case["kind"]
    if kind in ("walk", "host", "batch", "grid-walk"):
        return "exact"          # fixed-point sums: the same integers whatever the launch or the order
    if kind == "metrics":
        return {"rel": 1e-12}   # double-precision sums over at most 1e6 pixels (4e-16 from exact() at 512 x 512)
    # single-precision walks: the terms' rounding, and the few photons per million whose path a rounding sends
    # another way. About four times the distances from exact(): 2e-4 (density gradients), 1.2e-4 (image of the
    # fit step, gradients 3e-5), 8e-6 (1e7-photon gradient)
    if kind.startswith("grid"):
        return {"rel": 8e-4}
    return {"rel": 5e-4 if kind == "fit" else 3e-5}


# ------------------------------------------------------------------ the same in 64 bits


def _f64(v):
    return torch.as_tensor(v, dtype=torch.float64, device="cuda")


def _philox(p, event, key):
    """Four uniforms of Philox4x32-10 for counters (p low, p high, event, 0): ((r >> 9) + 1/2) 2^-23."""
    mask = 0xFFFFFFFF
    c = [p & mask, (p >> 32) & mask, torch.full_like(p, event & mask), torch.zeros_like(p)]
    k0, k1 = key & mask, (key >> 32) & mask
    for _ in range(10):
        a, b = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [((b >> 32) & mask) ^ c[1] ^ k0, b & mask, ((a >> 32) & mask) ^ c[3] ^ k1, a & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return [((r >> 9).double() + 0.5) * 2.0 ** -23 for r in c]


@functools.lru_cache(maxsize=64)
def _mie_levels(diameter_um, n_bins):
    """1 - cos theta at the levels i / n_bins of the Mie phase function's cumulative distribution in cos theta."""
    x, m = math.pi * diameter_um * 1e3 * N_MEDIUM / WAVELENGTH_NM, N_PARTICLE / N_MEDIUM
    n_max = int(x + 4.05 * x ** (1 / 3) + 10)
    d = np.zeros(int(max(n_max, m * x)) + 40)           # logarithmic derivative of psi_n(mx), downward
    for n in range(len(d) - 1, 0, -1):
        d[n - 1] = n / (m * x) - 1.0 / (d[n] + n / (m * x))
    fine = 1 << 17
    theta = torch.linspace(math.pi, 0.0, fine + 1, dtype=torch.float64, device="cuda")
    mu = torch.cos(theta)
    s1 = torch.zeros(fine + 1, dtype=torch.complex128, device="cuda")
    s2 = s1.clone()
    p0, p1 = torch.zeros_like(mu), torch.ones_like(mu)  # pi_{n-1}, pi_n
    psi0, psi1, chi0, chi1 = math.cos(x), math.sin(x), -math.sin(x), math.cos(x)
    for n in range(1, n_max + 1):
        psi, chi = (2 * n - 1) * psi1 / x - psi0, (2 * n - 1) * chi1 / x - chi0
        xi, xi1 = complex(psi, -chi), complex(psi1, -chi1)
        ta, tb = d[n] / m + n / x, m * d[n] + n / x
        a, b = (ta * psi - psi1) / (ta * xi - xi1), (tb * psi - psi1) / (tb * xi - xi1)
        f = (2 * n + 1) / (n * (n + 1.0))
        t = n * mu * p1 - (n + 1) * p0
        s1 += f * (a * p1 + b * t)
        s2 += f * (a * t + b * p1)
        p0, p1 = p1, ((2 * n + 1) * mu * p1 - (n + 1) * p0) / n
        psi0, psi1, chi0, chi1 = psi1, psi, chi1, chi
    dens = (s1.abs() ** 2 + s2.abs() ** 2) * torch.sin(theta)
    h = math.pi / fine
    f0, f1, f2 = dens[0:-1:2], dens[1::2], dens[2::2]
    cum = torch.cat([_f64([0.0]), torch.cumsum(h / 3 * (f0 + 4 * f1 + f2), 0)])
    want = cum[-1] * torch.arange(1, n_bins, device="cuda", dtype=torch.float64) / n_bins
    j = (torch.searchsorted(cum, want, right=True) - 1).clamp(0, fine // 2 - 1)
    rest, lo = want - cum[j], torch.zeros_like(want)
    hi = torch.full_like(want, 2 * h)
    c1, c2 = (-3 * f0 + 4 * f1 - f2)[j] / (4 * h), (f0 - 2 * f1 + f2)[j] / (6 * h * h)
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        low = mid * (f0[j] + mid * (c1 + mid * c2)) < rest
        lo, hi = torch.where(low, mid, lo), torch.where(low, hi, mid)
    th = math.pi - (2 * j.double() * h + lo)
    return torch.cat([_f64([2.0]), 2 * torch.sin(0.5 * th) ** 2, _f64([0.0])])


def _hat(mu, n_w):
    t = ((mu + 1.0) * (0.5 * (n_w - 1))).clamp(0.0, float(n_w - 1))
    k = t.floor().clamp(max=n_w - 2).long()
    return k, t - k


def _hat_integrals(om, n_w):
    """(breaks, density) of a table's pieces between its levels and the hat nodes, as 1 - cos theta descending,
    and the integrals of density times hat k."""
    n = om.numel() - 1
    nodes = 2.0 - 2.0 * torch.arange(n_w, device="cuda", dtype=torch.float64) / (n_w - 1)
    b = torch.unique(torch.cat([om, nodes])).flip(0)
    mid = 0.5 * (b[:-1] + b[1:])
    j = n - torch.searchsorted(om.flip(0).contiguous(), mid)
    j = j.clamp(0, n - 1)
    p = (1.0 / n) / (om[j] - om[j + 1])
    k, f = _hat(1.0 - mid, n_w)       # hats are linear on a piece: their mean is the value at its middle
    m = p * (b[:-1] - b[1:])
    z = torch.zeros(n_w, dtype=torch.float64, device="cuda")
    z.index_add_(0, k, m * (1 - f)).index_add_(0, k + 1, m * f)
    return b, p, z


def _weighted_levels(om, w):
    """Levels of the density p h_w / Z(w): its cumulative distribution inverted piece by piece (quadratic)."""
    n, n_w = om.numel() - 1, w.numel()
    b, p, _ = _hat_integrals(om, n_w)
    mid = 0.5 * (b[:-1] + b[1:])
    slope_k, _ = _hat(1.0 - mid, n_w)
    at = lambda v: w[slope_k] + (w[slope_k + 1] - w[slope_k]) * ((2.0 - v) * 0.5 * (n_w - 1) - slope_k)  # noqa: E731
    ha, hb, width = at(b[:-1]), at(b[1:]), b[:-1] - b[1:]
    cum = torch.cat([_f64([0.0]), torch.cumsum(p * 0.5 * (ha + hb) * width, 0)])
    want = cum[-1] * torch.arange(1, n, device="cuda", dtype=torch.float64) / n
    q = (torch.searchsorted(cum, want, right=True) - 1).clamp(0, p.numel() - 1)
    rem, s = (want - cum[q]) / p[q], ((hb - ha) / width)[q]
    x = 2 * rem / (ha[q] + torch.sqrt((ha[q] ** 2 + 2 * s * rem).clamp(min=0.0)))
    return torch.cat([_f64([2.0]), b[q] - x, _f64([0.0])])


def _camera_density(om, dy):
    """Phase density per steradian toward the camera: a table's bins (om: levels), or H-G (om None)."""
    if om is None:
        return (1 - HG_G ** 2) / (4 * math.pi) * ((1 - HG_G) ** 2 + 2 * HG_G * (1 - dy)) ** -1.5
    n = om.numel() - 1
    j = (n - torch.searchsorted(om.flip(0).contiguous(), (1.0 - dy).clamp(0.0, 2.0))).clamp(0, n - 1)
    return (1.0 / n) / (om[j] - om[j + 1]) / (2 * math.pi)


def _turned(d, om, u1, u2):
    """(new directions, 1 - cos theta): polar angle from u1, azimuth 2 pi u2 about d in the basis of Duff et al. (2017)."""
    if om is None:
        q = 1 - HG_G + 2 * HG_G * u1
        o = 2 * (1 - HG_G) ** 2 * (1 - u1) * (1 + HG_G * u1) / (q * q)
    else:
        t = u1 * (om.numel() - 1)
        i = t.long()
        o = om[i] + (t - i) * (om[i + 1] - om[i])
    dx, dy, dz = d
    st = torch.sqrt((o * (2 - o)).clamp(min=0.0))
    cp, sp = st * torch.cos(2 * math.pi * u2), st * torch.sin(2 * math.pi * u2)
    sg = torch.where(torch.signbit(dz), -1.0, 1.0).double()
    a = -1.0 / (sg + dz)
    b = dx * dy * a
    v = [(1 - o) * dx + cp * (1 + sg * dx * dx * a) + sp * b, (1 - o) * dy + cp * sg * b + sp * (sg + dy * dy * a),
         (1 - o) * dz - cp * sg * dx - sp * dy]
    r = torch.rsqrt(v[0] ** 2 + v[1] ** 2 + v[2] ** 2)
    return [c * r for c in v], o


def _entry(p, seed, radius):
    z = torch.zeros(p.numel(), dtype=torch.float64, device="cuda")
    pos, d = [z.clone(), z.clone(), z.clone()], [z + 1, z.clone(), z.clone()]
    if radius > 0:
        b = _philox(p, 0xFFFFFFFF, seed)
        rho = radius * torch.sqrt(b[0])
        pos[1], pos[2] = rho * torch.cos(2 * math.pi * b[1]), rho * torch.sin(2 * math.pi * b[1])
    return pos, d


def _cell(r, n, length, centred):
    return torch.floor(r * (n / length) + (0.5 * n if centred else 0.0)).long().clamp(0, n - 1)


def _survive(w, u, threshold, survival):
    """Weights after roulette (0: ended)."""
    low = w < threshold
    return torch.where(low, torch.where(u < survival, w / max(survival, 1e-300), torch.zeros_like(w)), w)


def _adjoint64(case, mu_s, mu_a, om, base, w_hat, adj, seed, image=None):
    """Value and gradients of sum(adj * image) for a homogeneous medium; adds the camera terms to `image` if given."""
    lx, ly, lz = case["lx"], case["ly"], case["lz"]
    nx, nz, n_w = case["nx"], case["nz"], case["n_w"]
    thr, surv = (1e-3, 0.0) if case["cut"] else (RR_THRESHOLD, RR_SURVIVAL)
    mu = mu_s + mu_a
    out = torch.zeros(3 + n_w, dtype=torch.float64, device="cuda")
    z = None
    if n_w:
        w_hat = torch.ones(n_w, dtype=torch.float64, device="cuda") if w_hat is None else w_hat
        z = _hat_integrals(base, n_w)[2]
        z = z / (w_hat * z).sum()
    chunk = 1_000_000
    for p0 in range(0, case["n"], chunk):
        m = min(chunk, case["n"] - p0)
        ph = torch.arange(m, device="cuda", dtype=torch.int64)
        pos, d = _entry(ph + p0, seed, case["beam_radius"])
        w, sc = torch.ones_like(pos[0]), torch.zeros_like(pos[0])
        run, angles, e = torch.zeros(m, dtype=torch.float64, device="cuda"), [], 0
        while ph.numel():
            u = _philox(ph + p0, e, seed)
            s = -torch.log(u[0]) / mu
            q = [s * a + r for a, r in zip(d, pos)]
            keep = (q[0] > 0) & (q[0] < lx) & (q[1].abs() < 0.5 * ly) & (q[2].abs() < 0.5 * lz)
            ph, w, sc, s = ph[keep], w[keep] * (mu_s / mu), sc[keep], s[keep]
            pos, d, u = [v[keep] for v in q], [v[keep] for v in d], [v[keep] for v in u]
            sc = sc + (1.0 / mu - s)
            e += 1
            ell = 0.5 * ly - pos[1]
            c = w * _camera_density(om, d[1]) * torch.exp(-mu * ell)
            pix = _cell(pos[2], nz, lz, True) * nx + _cell(pos[0], nx, lx, False)
            if image is not None:
                image.index_add_(0, pix, c)
            a = adj[pix] * c
            run[ph] += a
            out[0] += a.sum()
            out[1] += (a * (sc + e * (1.0 / mu_s - 1.0 / mu) - ell)).sum()
            out[2] += (a * (sc - e / mu - ell)).sum()
            if n_w:
                k, f = _hat(d[1], n_w)
                v = a / (w_hat[k] + f * (w_hat[k + 1] - w_hat[k]))
                out[3:].index_add_(0, k, v * (1 - f)).index_add_(0, k + 1, v * f)
                out[3:] -= e * a.sum() * z
            d, o = _turned(d, om, u[1], u[2])
            if n_w:
                angles.append((ph, 1.0 - o, run[ph].clone()))
            w = _survive(w, u[3], thr, surv)
            go = w > 0
            ph, w, sc, pos, d = ph[go], w[go], sc[go], [v[go] for v in pos], [v[go] for v in d]
        for i, mu_i, before in angles:
            k, f = _hat(mu_i, n_w)
            v = (run[i] - before) / (w_hat[k] + f * (w_hat[k + 1] - w_hat[k]))
            out[3:].index_add_(0, k, v * (1 - f)).index_add_(0, k + 1, v * f)
    return out


def _flight(maj, cells, size, lengths, tau, pos, d):
    """Delta-tracking flights through majorant cells (maj [mz, my, mx]): (hit, end points, majorant there)."""
    mz, my, mx = maj.shape
    dims, low = (mx, my, mz), (0.0, -0.5 * lengths[1], -0.5 * lengths[2])
    c = [_cell(pos[a], cells[a], lengths[a], a > 0).clone() for a in range(3)]
    c = [torch.div(c[a], size[a], rounding_mode="floor") for a in range(3)]
    vox = [lengths[a] / cells[a] for a in range(3)]
    inf = torch.full_like(tau, math.inf)

    def plane(a):
        i = torch.where(d[a] > 0, c[a] + 1, c[a])
        at = torch.clamp(i * size[a], max=cells[a]).double() * vox[a] + low[a]
        return torch.where(d[a] != 0, ((at - pos[a]) / d[a]).clamp(min=0.0), inf)

    t0, left = torch.zeros_like(tau), tau.clone()
    t = torch.stack([plane(a) for a in range(3)])
    done, hit = torch.zeros_like(tau, dtype=torch.bool), torch.zeros_like(tau, dtype=torch.bool)
    end, mb_end = torch.zeros_like(tau), torch.zeros_like(tau)
    while not bool(done.all()):
        flat = (c[2].clamp(0, mz - 1) * my + c[1].clamp(0, my - 1)) * mx + c[0].clamp(0, mx - 1)
        mb = maj.reshape(-1)[flat]
        t1, ax = t.min(0)
        t1 = torch.maximum(t1, t0)
        stop = ~done & (mb * (t1 - t0) > left)
        end = torch.where(stop, t0 + left / mb, end)
        mb_end = torch.where(stop, mb, mb_end)
        hit |= stop
        done = done | stop
        left = torch.where(done, left, left - mb * (t1 - t0))
        t0 = torch.where(done, t0, t1)
        for a in range(3):
            go = ~done & (ax == a)
            c[a] = torch.where(go, torch.where(d[a] > 0, c[a] + 1, c[a] - 1), c[a])
            out = go & ((c[a] < 0) | (c[a] >= dims[a]))
            done = done | out
            t[a] = torch.where(go, torch.maximum(plane(a), t0), t[a])
    return hit, [r + end * v for r, v in zip(pos, d)], mb_end


def _add_lengths(grad, coef, a, b, cells, lengths):
    """grad[voxel] += coef * length of the straight piece from a to b inside each voxel."""
    low = (0.0, -0.5 * lengths[1], -0.5 * lengths[2])
    for i in range(0, coef.numel(), 60_000):
        k = slice(i, i + 60_000)
        p, v = [x[k] for x in a], [y[k] - x[k] for x, y in zip(a, b)]
        ts = [torch.zeros_like(p[0])[:, None], torch.ones_like(p[0])[:, None]]
        for ax in range(3):
            planes = torch.arange(1, cells[ax], device="cuda", dtype=torch.float64) * (lengths[ax] / cells[ax]) + low[ax]
            t = (planes[None, :] - p[ax][:, None]) / torch.where(v[ax] == 0, torch.full_like(v[ax], 1e-300), v[ax])[:, None]
            ts.append(t.clamp(0.0, 1.0))
        t = torch.sort(torch.cat(ts, 1), 1)[0]
        mid, piece = 0.5 * (t[:, 1:] + t[:, :-1]), t[:, 1:] - t[:, :-1]
        at = [_cell(p[ax][:, None] + mid * v[ax][:, None], cells[ax], lengths[ax], ax > 0) for ax in range(3)]
        norm = torch.sqrt(v[0] ** 2 + v[1] ** 2 + v[2] ** 2)
        use = piece > 0
        idx = ((at[2] * cells[1] + at[1]) * cells[0] + at[0])[use]
        grad.index_add_(0, idx, ((coef[k] * norm)[:, None] * piece)[use])


def _grid_adjoint64(case, seed, density, adj, om):
    """Value and density gradient of sum(adj * image) for the voxel grid, exact lengths or null-collision scores."""
    cells, size, lengths = (case["gx"], case["gy"], case["gz"]), (case["bx"], case["by"], case["bz"]), (45.0, 10.0, 10.0)
    gx, gy, gz = cells
    mu = (K_EXT * density.double() + case["mu_a"])
    vy = 10.0 / gy
    above = (mu.flip(1).cumsum(1).flip(1) - mu) * vy
    pad = [(-g) % s for g, s in zip(cells, size)]
    m = torch.nn.functional.pad(mu, (0, pad[0], 0, pad[1], 0, pad[2]))
    mx, my, mz = [(g + s - 1) // s for g, s in zip(cells, size)]
    maj = m.reshape(mz, size[2], my, size[1], mx, size[0]).amax((1, 3, 5)) * (case["nulls"] or 1.0)
    grad = torch.zeros(gz * gy * gx, dtype=torch.float64, device="cuda")
    source = torch.zeros_like(grad)
    value, muf, abf = 0.0, mu.reshape(-1), above.reshape(-1)
    for p0 in range(0, case["n"], 250_000):
        n = min(250_000, case["n"] - p0)
        ph = torch.arange(n, device="cuda", dtype=torch.int64)
        pos, d = _entry(ph + p0, seed, 0.0)
        last = [v.clone() for v in pos]
        w = torch.ones(n, dtype=torch.float64, device="cuda")
        run, real, null, e = torch.zeros(n, dtype=torch.float64, device="cuda"), [], [], 0
        while ph.numel():
            u = _philox(ph + p0, e, seed)
            e += 1
            hit, end, mb = _flight(maj, cells, size, lengths, -torch.log(u[0]), pos, d)
            ph, w, mb, pos = ph[hit], w[hit], mb[hit], [v[hit] for v in end]
            d, last, u = [v[hit] for v in d], [v[hit] for v in last], [v[hit] for v in u]
            iy = _cell(pos[1], gy, 10.0, True)
            vox = (_cell(pos[2], gz, 10.0, True) * gy + iy) * gx + _cell(pos[0], gx, 45.0, False)
            acc = muf[vox] / mb
            r = u[3] < acc
            if case["nulls"]:
                x = ~r
                null.append((ph[x], vox[x], -K_EXT / (mb[x] - muf[vox[x]]), run[ph[x]].clone()))
            i, v, q = ph[r], vox[r], [c[r] for c in pos]
            wr = w[r] * case["albedo"] * (1.0 - case["mu_a"] / muf[v])
            top = (iy[r] + 1).double() * vy - 5.0
            cam = wr * _camera_density(om, d[1][r]) * torch.exp(-(muf[v] * (top - q[1]) + abf[v]))
            pix = _cell(q[2], case["nz"], 10.0, True) * case["nx"] + _cell(q[0], case["nx"], 45.0, False)
            a = adj[pix] * cam
            real.append((i, v, run[i].clone(), [c[r] for c in last], q))
            grad.index_add_(0, v, -K_EXT * a * (top - q[1]))
            source.index_add_(0, v, a)
            run[i] += a
            nd, _ = _turned([c[r] for c in d], om, u[1][r], u[2][r])
            for c, x in zip(d, nd):
                c[r] = x
            for c, x in zip(last, q):
                c[r] = x
            w[r] = _survive(wr, u[3][r] / acc[r], RR_THRESHOLD, RR_SURVIVAL)
            go = w > 0
            ph, w, pos, d, last = ph[go], w[go], [c[go] for c in pos], [c[go] for c in d], [c[go] for c in last]
        value += float(run.sum())
        for i, v, before, a, b in real:
            rest = run[i] - before
            grad.index_add_(0, v, rest * K_EXT / (muf[v] - case["mu_a"]))
            if not case["nulls"]:
                _add_lengths(grad, -K_EXT * rest, a, b, cells, lengths)
        for i, v, score, before in null:
            grad.index_add_(0, v, (run[i] - before) * score)
    s = source.reshape(gz, gy, gx)
    grad = grad.reshape(gz, gy, gx) - K_EXT * vy * (s.cumsum(1) - s)
    return _f64([value]), grad


def _metrics64(images, n_r):
    """Min-max normalised comparison of images 1, 2 with image 0, as image_metrics lays it out."""
    im = [i.double() for i in images]
    im = [(i - i.min()) / (i.max() - i.min()) for i in im]
    nz, nx = im[0].shape
    z = torch.arange(nz, device="cuda", dtype=torch.float64)[:, None] + 0.5 - nz / 2
    x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :] + 0.5 - nx / 2
    ring = torch.floor(torch.sqrt(x * x + z * z) / math.hypot(nx / 2, nz / 2) * n_r).long().clamp(max=n_r - 1).reshape(-1)
    count = torch.bincount(ring, minlength=n_r).double()
    has = count > 0
    prof = [torch.zeros(n_r, dtype=torch.float64, device="cuda").index_add_(0, ring, i.reshape(-1)) / count.clamp(min=1)
            for i in im]
    angle = 180.0 * (torch.arange(n_r, device="cuda") + 0.5) / n_r
    zones = [has & (angle < 30), has & (angle >= 30) & (angle <= 120), has & (angle > 120)]

    def pearson(a, b):
        a, b = a - a.mean(), b - b.mean()
        v = (a * a).sum() * (b * b).sum()
        return float((a * b).sum() / torch.sqrt(v)) if v > 0 else 0.0

    out = []
    for k in (1, 2):
        out += [float(((im[k] - im[0]) ** 2).mean().sqrt()), pearson(im[k], im[0])]
        out += [float(((prof[k] - prof[0])[q] ** 2).mean().sqrt()) if bool(q.any()) else 0.0 for q in zones]
        out.append(pearson(prof[k][has], prof[0][has]))
    closer = has & ((prof[1] - prof[0]).abs() < (prof[2] - prof[0]).abs())
    out.append(float(closer.sum() / has.sum()))
    return np.concatenate([np.array(out)] + [p.cpu().numpy() for p in prof])


def exact(case, seed):
    kind = case["kind"]
    if kind == "metrics":
        return _metrics64(prepare(case, seed)["images"], case["n_r"])
    if kind == "adjoint":
        mu_s, mu_a = _coefficients(case, seed)
        base = None if case["phase"] == "hg" else _mie_levels(case["diameter_um"], case["n_bins"])
        w = _weights(case, seed) if case["n_w"] else None
        om = _weighted_levels(base, w) if w is not None else base
        return _adjoint64(case, mu_s, mu_a, om, base, w, _adjoint_image(case, seed).double().reshape(-1), seed)
    if kind == "fit":
        mu_s, mu_a = _coefficients(case, seed)
        base = _mie_levels(case["diameter_um"], case["n_bins"])
        w = _weights(case, seed) if case["n_w"] else None
        om = _weighted_levels(base, w) if w is not None else base
        adj = _adjoint_image(case, seed).double().reshape(-1)
        image = torch.zeros(case["nz"] * case["nx"], dtype=torch.float64, device="cuda")
        _adjoint64(dict(case, n_w=0), mu_s, mu_a, om, base, None, adj, seed, image)
        g = _adjoint64(case, mu_s, mu_a, om, base, w, adj, seed + 1)
        return [image.reshape(case["nz"], case["nx"]), g[1], g[2]] + ([g[3:]] if w is not None else [])
    if kind in ("grid-grad", "grid-step"):
        # exact lengths through many voxels take a sort of every crossing: too long for the largest grids and budgets
        if not case["nulls"] and case["n"] * _steps(case["tau"]) * (case["gx"] + case["gy"] + case["gz"]) > 2.5e10:
            return None
        v, g = _grid_adjoint64(case, seed, _density(case, seed), _adjoint_image(case, seed).double().reshape(-1),
                               _mie_levels(5.0, 4096))
        return ([None, None, None] if kind == "grid-step" else []) + [v, g]
    return None     # fixed-point integers, compared exactly
