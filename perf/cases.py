"""Workloads of the MAR-DEAM library, one pass each through the public binding.

A case is one scan (or a batch of scans) and one call on it:
  iterate      Deam.iterate: MAR-DEAM iterations from a starting image
  gradient     Deam.gradient: the objective and its gradient
  autograd     i_divergence(c, deam) and its backward pass
  forward      Deam.forward: line integrals and expected counts
  backproject  Deam.backproject: the projector's adjoint
  init         Deam.mar_init: NMAR + FBP + decomposition with the user's prior
  batch        DeamBatch.iterate: uneven scans iterated together
The scanner is the one of the repository's tests and benchmark (SID 570 mm,
SDD 1040 mm, 0.75 mm rows at the isocentre, 90 and 140 kVp); measurements are
simulated here from exact chord lengths, so that they depend on the seed alone.
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

SID, SDD = 570.0, 1040.0
FAN2D, HELICAL = 0, 1
# an exact() pass over more Joseph samples than this is left out
EXACT_SAMPLES = 3.0e10

_BASE = dict(call="iterate", n_iter=1, nx=128, ny=128, nz=1, dx=0.98, dz=0.75, rows=1, row_mm=0.75, channels=256,
             per_rotation=360, rotations=1.0, pitch=0.6, bin_keV=1.0, i0=1e5, noise=0.0, metal="titanium",
             mask="ray", bowtie=False, clamp=False, lam=0.0, delta=0.05, start=0.3)


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one gradient of a 50 x 50 test slice, as a line search or a unit test makes it
        _case("slice50_gradient", call="gradient", nx=50, ny=50, dx=4.8, channels=70, per_rotation=64),
        # a whole small reconstruction: 10 iterations of a 128 x 128 fan-beam slice with a titanium disk
        _case("slice128_iterate", n_iter=10, nx=128, ny=128, dx=250.0 / 128, channels=256, per_rotation=360),
        # a clinical-size fan-beam slice at full angular sampling
        _case("slice512_iterate", n_iter=2, nx=512, ny=512, dx=0.6, channels=816, per_rotation=1160, bin_keV=2.0),
        # forward model of a ragged helical slab: line integrals and counts, as in data checks and calibration
        _case("slab_ragged_forward", call="forward", nx=301, ny=277, nz=37, dz=1.0, rows=15, channels=611,
              per_rotation=583, rotations=1.5, pitch=0.8, bin_keV=2.0, bowtie=True),
        # the adjoint alone on a ragged slab: the transpose that gradient solvers build on
        _case("slab_ragged_backproject", call="backproject", nx=277, ny=301, nz=45, rows=16, channels=701,
              per_rotation=720, rotations=1.5, pitch=0.8),
        # an ordinary slab with a bowtie, separate traces per spectrum and the nonnegativity option
        _case("slab384_iterate", nx=384, ny=384, nz=48, rows=16, channels=816, per_rotation=900, rotations=1.5,
              pitch=0.8, bin_keV=2.0, mask="per_spectrum", bowtie=True, clamp=True),
        # regularised MAR-DEAM on a thin slab
        _case("slab256_regularised", nx=256, ny=256, nz=16, dz=1.0, rows=16, channels=816, per_rotation=720,
              rotations=2.0, pitch=0.8, bin_keV=2.0, lam=5e3, delta=0.02),
        # plain 3D helical scan, slices twice as thick as the rows
        _case("helical256_iterate", nx=256, ny=256, nz=32, dz=1.5, rows=16, channels=672, per_rotation=1160,
              rotations=3.0, pitch=0.5, bin_keV=2.0, i0=2e5),
        # differentiation: forward and backward pass of the objective through autograd
        _case("helical256_autograd", call="autograd", nx=256, ny=256, nz=32, dz=1.5, rows=16, channels=672,
              per_rotation=1160, rotations=3.0, pitch=0.5, bin_keV=2.0, i0=2e5),
        # the starting image of a reconstruction, from a prior that the user has
        _case("helical256_init", call="init", nx=256, ny=256, nz=32, dz=1.5, rows=16, channels=672,
              per_rotation=1160, rotations=3.0, pitch=0.5, bin_keV=2.0, i0=2e5),
        # a worklist: uneven slices and slabs iterated together
        _case("batch8_iterate", call="batch", scans=8, sizes=7, bin_keV=2.0),
        # the full-size helical scan with steel hip inserts and electronic noise
        _case("helical512_iterate", nx=512, ny=512, nz=64, rows=16, channels=816, per_rotation=1160, rotations=5.0,
              pitch=0.6, noise=5.0, metal="steel"),
    ]


def _log(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def draw(rng):
    """One more case: a slice, a slab or a batch with sizes spread over the listed ranges."""
    kind = rng.choice(["slice", "slab", "slab", "slab", "batch"])
    if kind == "batch":
        return _case(call="batch", scans=rng.randint(2, 8), sizes=rng.randrange(1 << 20), bin_keV=2.0,
                     n_iter=rng.randint(1, 3))
    opts = dict(bin_keV=rng.choice([1.0, 2.0, 4.0]), metal=rng.choice(["titanium", "steel"]),
                mask=rng.choice(["ray", "ray", "per_spectrum", "none"]), bowtie=rng.random() < 0.4,
                clamp=rng.random() < 0.3, noise=rng.choice([0.0, 5.0]), start=round(rng.uniform(0.0, 6.2), 3))
    if kind == "slice":
        n = int(_log(rng, 40, 512))
        return _case(call=rng.choice(["iterate", "iterate", "gradient", "autograd", "forward", "backproject"]),
                     n_iter=rng.randint(1, 10), nx=n, ny=max(32, n - rng.randint(0, 24)),
                     dx=round(rng.uniform(240.0, 320.0) / n, 4), channels=int(n * rng.uniform(1.3, 2.0)),
                     per_rotation=int(_log(rng, 64, 1160)), **opts)
    nx = int(_log(rng, 96, 512))
    nz = int(_log(rng, 8, 64))
    dz = rng.choice([0.75, 1.0, 1.5])
    call = rng.choice(["iterate", "iterate", "regularised", "gradient", "autograd", "forward", "backproject", "init"])
    reg = dict(lam=round(_log(rng, 5e2, 1e4), 1), delta=0.02) if call == "regularised" else {}
    return _case(call="iterate" if reg else call, nx=nx, ny=max(80, nx - rng.randint(0, 40)), nz=nz, dz=dz,
                 rows=rng.choice([4, 11, 15, 16, 16, 16]), channels=int(_log(rng, 300, 816)),
                 per_rotation=int(_log(rng, 180, 1160)), rotations=rng.choice([1.0, 1.5, 2.0]),
                 pitch=rng.choice([0.5, 0.6, 0.8]), **reg, **opts)


def _batch_scans(case):
    """The scans of a batch: half fan-beam slices, half helical slabs of 16 slices or more."""
    rng = random.Random(case["sizes"])
    scans = []
    for i in range(case["scans"]):
        common = dict(n_iter=case["n_iter"], bin_keV=case["bin_keV"], metal=rng.choice(["titanium", "steel"]),
                      start=round(rng.uniform(0.0, 6.2), 3))
        if i % 2 == 0:
            n = rng.choice([128, 192, 256, 320, 384, 448, 512])
            scans.append(_case(nx=n, ny=n, dx=round(rng.uniform(240.0, 320.0) / n, 4), channels=8 * round(0.2 * n),
                               per_rotation=rng.randint(180, 1160), **common))
        else:
            n = rng.choice([256, 384])
            scans.append(_case(nx=n, ny=n, nz=rng.choice([16, 32]), dz=rng.choice([0.75, 1.0, 1.5]), rows=16,
                               channels=816, per_rotation=rng.randint(180, 720), rotations=2.0, pitch=0.8, **common))
    return scans


# ---- the scan: geometry, tables ---------------------------------------------

def _geometry(c):
    fov = max(c["nx"], c["ny"]) * c["dx"]
    flat = c["rows"] == 1
    views = int(round(c["per_rotation"] * c["rotations"]))
    feed = 0.0 if flat else c["pitch"] * c["rows"] * c["row_mm"]
    return SimpleNamespace(
        kind=FAN2D if flat else HELICAL, nx=c["nx"], ny=c["ny"], nz=c["nz"], dx=c["dx"], dy=c["dx"], dz=c["dz"],
        cx=0.0, cy=0.0, cz=0.0, sid=SID, sdd=SDD, n_views=views, views_per_rotation=c["per_rotation"],
        start_angle=c["start"], feed=feed, z_start=-feed * views / c["per_rotation"] / 2.0, n_rows=c["rows"],
        row_pitch=1.0 if flat else c["row_mm"] * SDD / SID, n_channels=c["channels"],
        channel_pitch=2.0 * math.asin(fov / 2.0 / SID) * 1.02 / c["channels"], channel_offset=0.25, row_offset=0.0)


# photoelectric and Compton parts of the attenuation at 60 keV, 1/mm
_MATERIALS = {"polystyrene": (0.0008, 0.0188), "cacl2": (0.0170, 0.0230), "aluminium": (0.0400, 0.0350),
              "titanium": (0.1700, 0.0550), "steel": (0.8400, 0.1100)}


def _klein_nishina(E):
    k = np.asarray(E, np.float64) / 510.998950
    lg = np.log1p(2 * k)
    return (1 + k) / k**2 * (2 * (1 + k) / (1 + 2 * k) - lg / k) + lg / (2 * k) - (1 + 3 * k) / (1 + 2 * k) ** 2


def _mu(material, E):
    photo, compton = _MATERIALS[material]
    return photo * (60.0 / E) ** 3 + compton * _klein_nishina(E) / _klein_nishina(60.0)


def _tables(c):
    n = int(round(120.0 / c["bin_keV"]))
    E = 20.0 + (np.arange(n) + 0.5) * c["bin_keV"]
    I0 = []
    for kvp, al in ((90.0, 2.5), (140.0, 6.0)):
        phi = np.clip(kvp - E, 0.0, None) * np.exp(-_mu("aluminium", E) * al)
        I0.append(phi * (c["i0"] / phi.sum()))
    bow = None
    if c["bowtie"]:
        x = (np.arange(c["channels"]) - (c["channels"] - 1) / 2.0) / c["channels"]
        bow = np.exp(-2.0 * x * x)
    return E, np.stack(I0), np.stack([_mu("polystyrene", E), _mu("cacl2", E)]), _mu(c["metal"], E), bow


# ---- the object and its measurement -----------------------------------------

def _objects(c, seed):
    """(centre, semi-axes, c1, c2, metal): elliptic body along z, seeded inserts, metal rods that displace tissue.
    A third semi-axis of None is a cylinder along z."""
    rng = random.Random(1000 + seed)
    a, b = 0.42 * c["nx"] * c["dx"], 0.32 * c["ny"] * c["dx"]
    objs = [((0.0, 0.0, 0.0), (a, b, None), 1.0, 0.02, 0.0)]
    half = c["nz"] * c["dz"] / 2.0
    for d1, d2 in ((-0.1, 0.45), (-0.3, 0.30), (-0.05, 0.15), (-0.08, 0.0)):
        phi, rho, r = rng.uniform(0, 2 * math.pi), rng.uniform(0.2, 0.6), rng.uniform(0.08, 0.16) * b
        z = rng.uniform(-0.5, 0.5) * half
        objs.append(((rho * a * math.cos(phi), rho * b * math.sin(phi), z),
                     (r, 0.8 * r, None if c["nz"] == 1 else 1.5 * r), d1, d2, 0.0))
    for side in (-1.0, 1.0):
        at, axes = (side * 0.45 * a, 0.05 * b, 0.0), (0.05 * b, 0.04 * b, None)
        objs.append((at, axes, -1.0, -0.02, 0.0))
        objs.append((at, axes, 0.0, 0.0, 1.0))
    return objs


def _angles(g, views, device):
    beta = g.start_angle + 2.0 * math.pi * views / g.views_per_rotation
    gam = (torch.arange(g.n_channels, device=device, dtype=torch.float64) - (g.n_channels - 1) / 2.0
           + g.channel_offset) * g.channel_pitch
    w = (torch.arange(g.n_rows, device=device, dtype=torch.float64) - (g.n_rows - 1) / 2.0 + g.row_offset) * g.row_pitch
    return beta, gam, w


def _paths(c, g, seed, views, device):
    """Basis and metal path lengths (mm) of every ray of the views, float32 [v, R, K]."""
    beta, gam, w = _angles(g, views, device)
    ang = beta[:, None] + gam[None, :]
    ux, uy = (-SDD * torch.cos(ang))[:, None, :], (-SDD * torch.sin(ang))[:, None, :]
    uz = w[None, :, None]
    sx, sy = (SID * torch.cos(beta))[:, None, None], (SID * torch.sin(beta))[:, None, None]
    sz = (g.z_start + g.feed * views / g.views_per_rotation)[:, None, None]
    norm = torch.sqrt(SDD * SDD + uz * uz)
    out = [torch.zeros((len(views), g.n_rows, g.n_channels), device=device) for _ in range(3)]
    for (ox, oy, oz), (a, b, h), d1, d2, m in _objects(c, seed):
        A = (ux / a) ** 2 + (uy / b) ** 2
        B = ux * (sx - ox) / a**2 + uy * (sy - oy) / b**2
        C = ((sx - ox) / a) ** 2 + ((sy - oy) / b) ** 2 - 1.0
        if h is not None:  # ellipsoid
            A = A + (uz / h) ** 2
            B = B + uz * (sz - oz) / h**2
            C = C + ((sz - oz) / h) ** 2
        L = (2.0 * torch.sqrt(torch.clamp(B * B - A * C, min=0.0)) / A * norm).float()
        for o, d in zip(out, (d1, d2, m)):
            if d:
                o.add_(L, alpha=d)
    return out


def _measure(c, g, seed, device):
    """Counts [2, V, R, K] (Poisson, optional electronic noise) and the metal path length [V, R, K]."""
    E, I0, mu, mum, bow = _tables(c)
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    shape = (g.n_views, g.n_rows, g.n_channels)
    d = torch.empty((2,) + shape, device=device)
    metal = torch.empty(shape, device=device)
    step = max(1, int(2e7 // (g.n_rows * g.n_channels)))
    for v0 in range(0, g.n_views, step):
        views = torch.arange(v0, min(g.n_views, v0 + step), device=device, dtype=torch.float64)
        l1, l2, lm = _paths(c, g, seed, views, device)
        sl = slice(v0, v0 + len(views))
        metal[sl] = lm
        counts = [torch.zeros_like(l1), torch.zeros_like(l1)]
        for e in range(len(E)):
            att = torch.exp_((l1 * -float(mu[0, e])).add_(l2, alpha=-float(mu[1, e])).add_(lm, alpha=-float(mum[e])))
            for j in range(2):
                if I0[j, e] > 0:
                    counts[j].add_(att, alpha=float(I0[j, e]))
        for j in range(2):
            x = counts[j]
            if bow is not None:
                x = x * torch.as_tensor(bow, dtype=torch.float32, device=device)
            x = torch.poisson(x, generator=gen)
            if c["noise"]:
                x = x + c["noise"] * torch.randn(x.shape, generator=gen, device=device)
            d[j, sl] = x
    return d, metal


def _images(c, g, seed, device):
    """A starting image [nz, ny, nx, 2] (soft tissue in the body, 1 % noise) and a prior [nz, ny, nx] in 1/mm."""
    gen = torch.Generator(device=device)
    gen.manual_seed(seed + 1)
    x = (torch.arange(g.nx, device=device) - (g.nx - 1) / 2.0) * g.dx
    y = (torch.arange(g.ny, device=device) - (g.ny - 1) / 2.0) * g.dy
    a, b = 0.42 * c["nx"] * c["dx"], 0.32 * c["ny"] * c["dx"]
    body = ((x / a) ** 2 + (y[:, None] / b) ** 2 <= 1.0).float().expand(g.nz, g.ny, g.nx)
    image = body[..., None] * torch.tensor([0.95, 0.05], device=device)
    image = image + 0.01 * body[..., None] * torch.rand(image.shape, generator=gen, device=device)
    prior = 0.0195 * body * (1.0 + 0.05 * torch.rand(body.shape, generator=gen, device=device))
    return image.contiguous(), prior.contiguous()


def _inputs(c, seed):
    """Everything a pass reads, on the GPU, from the seed alone."""
    device = torch.device("cuda")
    g = _geometry(c)
    s = SimpleNamespace(case=c, geo=g, tables=_tables(c))
    s.image, s.prior = _images(c, g, seed, device)
    if c["call"] == "backproject":
        gen = torch.Generator(device=device)
        gen.manual_seed(seed)
        s.rays = torch.rand((g.n_views, g.n_rows, g.n_channels, 2), generator=gen, device=device)
        return s
    if c["call"] == "forward":
        return s
    s.counts, metal = _measure(c, g, seed, device)
    t = 0.5 * min(g.dx, g.dz) if g.nz > 1 else 0.5 * g.dx
    s.trace = None
    if c["mask"] == "ray":
        s.trace = (metal >= t).to(torch.uint8)
    elif c["mask"] == "per_spectrum":
        s.trace = torch.stack([metal >= t, metal >= 2.0 * t]).to(torch.uint8)
    return s


_CALIB = (0.0256, 0.0530, 0.0196, 0.0290)  # Eq. (4) weights of a typical scan of these spectra


def _scan(c, seed):
    import paper_2202_00116_gb300 as pkg
    s = _inputs(c, seed)
    E, I0, mu, _, bow = s.tables
    s.deam = pkg.Deam(s.geo, I0, mu, bowtie=bow, energies=E, clamp_nonneg=c["clamp"], penalty_lambda=c["lam"],
                      penalty_delta=c["delta"])
    if hasattr(s, "counts"):
        s.deam.set_data(s.counts)
        if s.trace is not None:
            s.deam.set_metal_mask(s.trace, c["mask"])
        s.counts = s.trace = None
    return s


def prepare(case, seed):
    import paper_2202_00116_gb300 as pkg
    if case["call"] != "batch":
        s = _scan(case, seed)
        if case["call"] == "autograd":
            s.image.requires_grad_(True)
        return s
    scans = [_scan(c, seed + 31 * i) for i, c in enumerate(_batch_scans(case))]
    return SimpleNamespace(case=case, scans=scans, work=[s.image.clone() for s in scans],
                           batch=pkg.DeamBatch([s.deam for s in scans]))


def run(state):
    import paper_2202_00116_gb300 as pkg
    c = state.case
    call = c["call"]
    if call == "iterate":
        image = state.image.clone()
        history = state.deam.iterate(image, c["n_iter"])
        return {"image": image, "objective": history.tolist()}
    if call == "gradient":
        grad, F = state.deam.gradient(state.image)
        return {"gradient": grad, "objective": F}
    if call == "autograd":
        state.image.grad = None
        F = pkg.i_divergence(state.image, state.deam)
        F.backward()
        return {"gradient": state.image.grad, "objective": float(F.detach())}
    if call == "forward":
        lines, counts = state.deam.forward(state.image, want_l=True, want_g=True)
        return {"lines": lines, "counts": counts}
    if call == "backproject":
        return {"image": state.deam.backproject(state.rays)}
    if call == "init":
        image, _, mu = state.deam.mar_init(_CALIB, t_air=0.005, t_bone=0.026, soft_value=0.0195, prior=state.prior)
        return {"image": image, "fbp": mu}
    for w, s in zip(state.work, state.scans):
        w.copy_(s.image)
    history = state.batch.iterate(state.work, c["n_iter"])
    return {"images": state.work, "objective": history.reshape(-1).tolist()}


def _samples(c):
    """Joseph samples of one projection: rays times planes, less what passes beside the volume."""
    g = _geometry(c)
    return 0.83 * g.n_views * g.n_rows * g.n_channels * max(g.nx, g.ny)


def work(case):
    if case["call"] == "batch":
        parts = [work(c) for c in _batch_scans(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    g, call = _geometry(case), case["call"]
    rays, vox, bins = g.n_views * g.n_rows * g.n_channels, g.nx * g.ny * g.nz, int(round(120.0 / case["bin_keV"]))
    # per sample: the forward blends 4 taps of 2 components, the adjoint spreads 4 (or 2) components to 4 taps
    fwd, adj, spectral = 16.0 * _samples(case), 32.0 * _samples(case), 17.0 * bins * rays
    data = 8 * rays + (rays if case["mask"] != "none" else 0)
    if call == "iterate":
        n = case["n_iter"]
        return {"bytes": n * (16 * vox + data), "flops": n * (fwd + adj + spectral)}
    if call == "gradient":
        return {"bytes": 16 * vox + data, "flops": fwd + adj / 2 + spectral}
    if call == "autograd":
        return {"bytes": 24 * vox + 2 * data, "flops": 2 * fwd + adj / 2 + 2 * spectral}
    if call == "forward":
        return {"bytes": 8 * vox + 16 * rays, "flops": fwd + 7.0 * bins * rays}
    if call == "backproject":
        return {"bytes": 8 * rays + 8 * vox, "flops": adj / 2}
    # both spectra filtered by FFT-sized work, one bilinear sample per voxel, view and spectrum; the prior projected once
    views = min(g.n_views, g.views_per_rotation)
    return {"bytes": data + 24 * vox, "flops": 2 * rays * 5 * math.log2(g.n_channels) + 2 * 10.0 * vox * views + fwd / 2}


# ---- 64-bit values of the outputs ---------------------------------------------

class _Exact:
    """Joseph's projector, Eq. (8) and the c-step in float64 with plain torch operations."""

    def __init__(self, s):
        self.c, self.g = s.case, s.geo
        self.dev = torch.device("cuda")
        g = self.g
        self.X0, self.Y0, self.Z0 = -(g.nx - 1) / 2.0 * g.dx, -(g.ny - 1) / 2.0 * g.dy, -(g.nz - 1) / 2.0 * g.dz
        _, I0, mu, _, bow = s.tables
        self.I0 = torch.as_tensor(I0, device=self.dev)
        self.mu = torch.as_tensor(mu, device=self.dev)
        self.bow = None if bow is None else torch.as_tensor(bow, device=self.dev)

    def chunks(self):
        """Rays of one dominant axis: (axis, views, channels, fq, t, length) with the last dimension the planes."""
        g = self.g
        step = max(1, int(2.5e7 // (g.n_channels * max(g.nx, g.ny))))
        for v0 in range(0, g.n_views, step):
            views = torch.arange(v0, min(g.n_views, v0 + step), device=self.dev, dtype=torch.float64)
            beta, gam, _ = _angles(g, views, self.dev)
            ang = beta[:, None] + gam[None, :]
            dx, dy = -torch.cos(ang), -torch.sin(ang)
            xdom = dx.abs() >= dy.abs()
            for axis in (0, 1):
                iv, ik = torch.nonzero(xdom if axis == 0 else ~xdom, as_tuple=True)
                if not len(iv):
                    continue
                sx = (SID * torch.cos(beta[iv]) - self.X0) / g.dx
                sy = (SID * torch.sin(beta[iv]) - self.Y0) / g.dy
                a, b = dx[iv, ik], dy[iv, ik]
                if axis == 0:
                    sp, sq, slope, kappa, L, n = sx, sy, b / a * g.dx / g.dy, g.dx / SDD / a, g.dx / a.abs(), g.nx
                else:
                    sp, sq, slope, kappa, L, n = sy, sx, a / b * g.dy / g.dx, g.dy / SDD / b, g.dy / b.abs(), g.ny
                p = torch.arange(n, device=self.dev, dtype=torch.float64)[None, :] - sp[:, None]
                sz = (g.z_start + g.feed * views[iv] / g.views_per_rotation - self.Z0) / g.dz
                yield axis, views[iv].long(), ik, sq[:, None] + p * slope[:, None], p * kappa[:, None], L, sz

    def taps(self, axis, fq, t, sz, r):
        """Selected samples of row r: (flat index into [rays, planes], padded voxel index, q weight, z weight, strides)."""
        g = self.g
        w = (r - (g.n_rows - 1) / 2.0 + g.row_offset) * g.row_pitch
        fz = sz[:, None] + (w / g.dz) * t
        nq = g.ny if axis == 0 else g.nx
        sel = torch.nonzero(((fq > -1) & (fq < nq) & (fz > -1) & (fz < g.nz)).reshape(-1)).squeeze(1)
        q, z = fq.reshape(-1)[sel], fz.reshape(-1)[sel]
        jq, jz = torch.floor(q), torch.floor(z)
        p = sel % fq.shape[1]
        row, plane = g.nx + 2, (g.ny + 2) * (g.nx + 2)
        sp, sq = (1, row) if axis == 0 else (row, 1)
        e = (jz.long() + 1) * plane + (p + 1) * sp + (jq.long() + 1) * sq
        return sel, e, q - jq, z - jz, sq, plane, math.sqrt(1.0 + (w / SDD) ** 2)

    def pad(self, img):
        return torch.nn.functional.pad(img, (0, 0, 1, 1, 1, 1, 1, 1)).reshape(-1, img.shape[-1])

    def forward(self, img):
        """l [V, R, K, n] of img [nz, ny, nx, n]."""
        g = self.g
        v = self.pad(img.double())
        out = torch.empty((g.n_views, g.n_rows, g.n_channels, v.shape[1]), dtype=torch.float64, device=self.dev)
        for axis, iv, ik, fq, t, L, sz in self.chunks():
            for r in range(g.n_rows):
                sel, e, wq, wz, sq, plane, rowf = self.taps(axis, fq, t, sz, r)
                wq, wz = wq[:, None], wz[:, None]
                val = torch.lerp(torch.lerp(v[e], v[e + sq], wq), torch.lerp(v[e + plane], v[e + plane + sq], wq), wz)
                dense = torch.zeros((fq.numel(), v.shape[1]), dtype=torch.float64, device=self.dev)
                dense[sel] = val
                out[iv, r, ik] = dense.reshape(fq.shape + (-1,)).sum(1) * (L * rowf)[:, None]
        return out

    def adjoint(self, y):
        """A^T y [nz, ny, nx, n] of y [V, R, K, n]."""
        g = self.g
        n = y.shape[-1]
        out = torch.zeros(((g.nz + 2) * (g.ny + 2) * (g.nx + 2), n), dtype=torch.float64, device=self.dev)
        for axis, iv, ik, fq, t, L, sz in self.chunks():
            for r in range(g.n_rows):
                sel, e, wq, wz, sq, plane, rowf = self.taps(axis, fq, t, sz, r)
                P = (y[iv, r, ik].double() * (L * rowf)[:, None])[sel // fq.shape[1]]
                for off, w in ((0, (1 - wq) * (1 - wz)), (sq, wq * (1 - wz)), (plane, (1 - wq) * wz),
                               (plane + sq, wq * wz)):
                    out.index_add_(0, e + off, P * w[:, None])
        return out.reshape(g.nz + 2, g.ny + 2, g.nx + 2, n)[1:-1, 1:-1, 1:-1].contiguous()

    def counts(self, l):
        """g [2, ...] and S [2 spectra, 2 components, ...] of line integrals l [..., 2]."""
        out = torch.zeros((2,) + l.shape[:-1], dtype=torch.float64, device=self.dev)
        S = torch.zeros((2, 2) + l.shape[:-1], dtype=torch.float64, device=self.dev)
        for e in range(self.mu.shape[1]):
            if not bool((self.I0[:, e] > 0).any()):
                continue
            x = torch.exp(-(l[..., 0] * self.mu[0, e] + l[..., 1] * self.mu[1, e]))
            for j in range(2):
                out[j].add_(x, alpha=float(self.I0[j, e]))
                for i in range(2):
                    S[j, i].add_(x, alpha=float(self.I0[j, e] * self.mu[i, e]))
        if self.bow is not None:
            out *= self.bow
            S *= self.bow
        return out, S

    def rays(self, s, img):
        """Payload (B1, B2, D1, D2) [V, R, K, 4] and the objective at img."""
        pay = torch.empty(s.counts.shape[1:] + (4,), dtype=torch.float64, device=self.dev)
        F = 0.0
        l = self.forward(img)
        step = max(1, int(1e7 // (self.g.n_rows * self.g.n_channels)))
        for v0 in range(0, self.g.n_views, step):
            sl = slice(v0, v0 + step)
            q, S = self.counts(l[sl])
            d = torch.clamp(s.counts[:, sl].double(), min=0.0)
            off = torch.ones_like(d)
            if s.trace is not None:
                off = (s.trace[:, sl] == 0).double() if s.trace.dim() == 4 else (s.trace[sl] == 0).double().expand_as(d)
            u = (d - q) / q * off
            pay[sl, ..., 0], pay[sl, ..., 1] = S[0, 0] + S[1, 0], S[0, 1] + S[1, 1]
            pay[sl, ..., 2], pay[sl, ..., 3] = u[0] * S[0, 0] + u[1] * S[1, 0], u[0] * S[0, 1] + u[1] * S[1, 1]
            F += float((off * (torch.special.xlogy(d, d / q) - d + q)).sum())
        return pay, F

    def normaliser(self):
        g = self.g
        active = (self.I0 > 0).any(0)
        h = self.forward(torch.ones((g.nz, g.ny, g.nx, 1), device=self.dev)).max()
        return float((self.mu[0] + self.mu[1])[active].max()) * float(h)

    def iterate(self, s, n_iter):
        img = s.image.double()
        Z, hist = self.normaliser(), []
        for _ in range(n_iter):
            pay, F = self.rays(s, img)
            hist.append(F)
            sums = self.adjoint(pay)
            bt, bh = sums[..., :2], sums[..., :2] + sums[..., 2:]
            if self.c["lam"] > 0:
                img = self.regularised(img, bt, bh, Z)
            else:
                ok = (bt > 0) & (bh > 0)
                step = torch.log1p(torch.where(ok, sums[..., 2:] / torch.where(ok, bt, 1.0), 0.0)) / Z
                new = torch.where(ok, img - step, img)
                img = torch.where(ok, torch.clamp(new, min=0.0), new) if self.c["clamp"] else new
        return img, hist

    def regularised(self, c, bt, bh, Z):
        """Per voxel and component the root of G'(t) = bh - bt e^(-Z (t - c)) + 2 lam sum_n w_n phi'(2 t - m_n)."""
        g, lam, delta = self.g, self.c["lam"], self.c["delta"]
        has = torch.ones((g.nz, g.ny, g.nx, 1), dtype=torch.float64, device=self.dev)
        pc, ph = (torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1)) for x in (c, has))
        m, w = [], []
        for oz in (-1, 0, 1):
            for oy in (-1, 0, 1):
                for ox in (-1, 0, 1):
                    if ox or oy or oz:
                        at = (slice(1 + oz, 1 + oz + g.nz), slice(1 + oy, 1 + oy + g.ny), slice(1 + ox, 1 + ox + g.nx))
                        m.append(c + pc[at])
                        w.append(ph[at] / math.sqrt((ox * g.dx) ** 2 + (oy * g.dy) ** 2 + (oz * g.dz) ** 2))
        seen = bt > 0
        keep = seen & ~(bh > 0)
        bt, bh = torch.where(seen, bt, 0.0), torch.where(seen, bh, 0.0)

        def slope(t):
            e = bt * torch.exp(-Z * (t - c))
            gp = bh - e
            for mn, wn in zip(m, w):
                u = 2 * t - mn
                a = 1 + u.abs() / delta
                gp = gp + 2 * lam * wn * u / a
            return gp

        lo, hi = c - 1.0, c + 1.0
        for _ in range(40):  # widen to a bracket
            a, b = slope(lo) > 0, slope(hi) < 0
            if not bool((a | b).any()):
                break
            lo, hi = torch.where(a, lo - (hi - lo), lo), torch.where(b, hi + (hi - lo), hi)
        for _ in range(60):  # G' increases: plain bisection, as Newton's step may cycle on the penalty's bend
            t = 0.5 * (lo + hi)
            up = slope(t) > 0
            hi, lo = torch.where(up, t, hi), torch.where(up, lo, t)
        new = torch.where(keep, c, t)
        return torch.clamp(new, min=0.0) if self.c["clamp"] else new

    # -- starting image: logarithm, NMAR completion, filtered backprojection, decomposition --
    def init(self, s):
        g = self.g
        i0 = self.I0.sum(1)[:, None, None, None]
        if self.bow is not None:
            i0 = i0 * self.bow
        p = torch.log(i0 / torch.clamp(s.counts.double(), min=1.0))
        if s.trace is not None:
            h = torch.clamp(self.forward(s.prior[..., None])[..., 0], min=1e-3)
            for j in range(2):
                on = (s.trace[j] if s.trace.dim() == 4 else s.trace) != 0
                p[j] = torch.where(on, self.interpolate(p[j] / h, on) * h, p[j])
        mu = self.fbp(p)
        M = torch.tensor(_CALIB, dtype=torch.float64, device=self.dev).reshape(2, 2)
        return torch.einsum("ij,j...->...i", torch.linalg.inv(M), mu), mu

    def interpolate(self, n, on):
        k = torch.arange(self.g.n_channels, device=self.dev).expand(on.shape)
        K = self.g.n_channels
        left = torch.where(on, -1, k).cummax(-1).values
        right = torch.where(on, K, k).flip(-1).cummin(-1).values.flip(-1)
        a, b = torch.gather(n, -1, left.clamp(min=0)), torch.gather(n, -1, right.clamp(max=K - 1))
        f = (k - left).double() / (right - left).clamp(min=1).double()
        val = torch.where(left < 0, b, torch.where(right >= K, a, a + (b - a) * f))
        return torch.where((left < 0) & (right >= K), n, val)

    def fbp(self, p):
        g, K = self.g, self.g.n_channels
        _, gam, w = _angles(g, torch.zeros(1, device=self.dev, dtype=torch.float64), self.dev)
        da = g.channel_pitch
        n = torch.arange(K, device=self.dev, dtype=torch.float64)
        ker = torch.where(n % 2 == 1, -1.0 / (2 * math.pi**2 * torch.sin(n * da) ** 2), 0.0)
        ker[0] = 1.0 / (8 * da * da)
        idx = torch.arange(K, device=self.dev)
        q = (p * (SID * torch.cos(gam)) * (SDD / torch.sqrt(SDD**2 + w * w))[:, None]) @ (
            da * ker[(idx[:, None] - idx[None, :]).abs()])
        x = (torch.arange(g.nx, device=self.dev, dtype=torch.float64) - (g.nx - 1) / 2.0) * g.dx
        y = (torch.arange(g.ny, device=self.dev, dtype=torch.float64) - (g.ny - 1) / 2.0) * g.dy
        out = torch.zeros((2, g.nz, g.ny, g.nx), dtype=torch.float64, device=self.dev)
        N, V, R = g.views_per_rotation, g.n_views, g.n_rows
        lo, hi = [], []
        for iz in range(g.nz):
            a, b = 0, min(V, N)
            if g.feed and R > 1:
                a = math.ceil((self.Z0 + iz * g.dz - g.z_start) * N / g.feed - N / 2.0)
                b = a + N
            lo.append(max(a, 0))
            hi.append(max(max(a, 0), min(b, V)))
        lo_t, hi_t = torch.tensor(lo, device=self.dev), torch.tensor(hi, device=self.dev)
        zs = self.Z0 + torch.arange(g.nz, device=self.dev, dtype=torch.float64) * g.dz
        for v in range(V):
            use = torch.nonzero((lo_t <= v) & (v < hi_t)).squeeze(1)
            if not len(use):
                continue
            beta = g.start_angle + 2 * math.pi * v / N
            cb, sb = math.cos(beta), math.sin(beta)
            ddx, ddy = (x - SID * cb)[None, :], (y - SID * sb)[:, None]
            L2 = ddx**2 + ddy**2
            kf = torch.atan2(ddx * sb - ddy * cb, -(ddx * cb + ddy * sb)) / da + (K - 1) / 2.0 - g.channel_offset
            inside = (kf >= 0) & (kf <= K - 1)
            k0 = kf.clamp(0, K - 2).floor().long().clamp(max=K - 2)
            ak = kf - k0
            rf = ((zs[use] - g.z_start - g.feed * v / N)[:, None, None] * SDD / torch.sqrt(L2) / g.row_pitch
                  + (R - 1) / 2.0 - g.row_offset).clamp(0, R - 1)
            r0 = rf.floor().long().clamp(max=max(R - 2, 0))
            ar = rf - r0 if R > 1 else torch.zeros_like(rf)
            at = r0 * K + k0
            up = K if R > 1 else 0
            for j in range(2):
                f = q[j, v].reshape(-1)
                val = torch.lerp(torch.lerp(f[at], f[at + 1], ak.expand_as(at)),
                                 torch.lerp(f[at + up], f[at + up + 1], ak.expand_as(at)), ar)
                out[j, use] += torch.where(inside, val / L2, 0.0)
        return out * (2 * math.pi / N)


def exact(case, seed):
    """run(prepare(case, seed)) in 64 bits; None where it would take long."""
    call = case["call"]
    if call == "batch":
        images, hist = [], []
        for i, c in enumerate(_batch_scans(case)):
            # the slices of the batch: its slabs are the kind of scan that the single cases cover
            got = exact(c, seed + 31 * i) if c["nz"] == 1 else None
            images.append(None if got is None else got["image"])
            hist += [None] * c["n_iter"] if got is None else got["objective"]
        return {"images": images, "objective": hist}
    passes = {"iterate": 2 * case["n_iter"], "gradient": 2, "autograd": 2}.get(call, 1)
    if passes * _samples(case) > EXACT_SAMPLES:
        return None
    s = _inputs(case, seed)
    X = _Exact(s)
    if call == "iterate":
        image, hist = X.iterate(s, case["n_iter"])
        return {"image": image, "objective": hist}
    if call in ("gradient", "autograd"):
        pay, F = X.rays(s, s.image)
        return {"gradient": X.adjoint(pay[..., 2:].contiguous()), "objective": F}
    if call == "forward":
        lines = X.forward(s.image)
        return {"lines": lines, "counts": X.counts(lines)[0]}
    if call == "backproject":
        return {"image": X.adjoint(s.rays)}
    image, mu = X.init(s)
    return {"image": image, "fbp": mu}
