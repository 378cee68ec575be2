"""The gather backprojection over its plans: every slab depth and number of view
groups that bwd_plan picks, ragged columns and slices, windows of many channels,
rows whose samples straddle slices, one row, one column, a volume off the axis.
The adjoint is compared with the oracle's, the fused c-step's sums with the
adjoint of the payload, the gradient with the sums; on the large volumes, where
FP32 ray positions (|q| up to 512 voxels) and white-noise rays of few views differ
element by element, with the forward kernel by the adjoint identity, to the bar
that the other adjoint identities have.

Tolerance of the adjoint, rel-L2 1e-5: the FP32 sample heights are rounded to
about 2e-6 slice at |z| < 64, which moves that share of a sample's weight from one
slice to the next, and sums of up to 1e4 terms round to about 2e-6; 1e-5 is the
bar that the projections have."""
import dataclasses

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2202_00116_gb300 import build
    build.build()
    import oracle
    oracle.build()
    import paper_2202_00116_gb300 as p
    return p


def _geo(**kw):
    """Helical geometry of the tests' scanner; fan and rows follow the sizes."""
    g = dict(nx=40, ny=36, nz=12, dx=4.0, dz=0.75, R=16, K=96, V=48, vpr=48, pitch=0.8, row_mm=0.75, start=0.3,
             cx=0.0, cy=0.0, cz=0.0, dy=None, row_offset=0.0, feed=2.0)
    g.update(kw)
    feed = g["pitch"] * g["R"] * g["row_mm"] if g["R"] > 1 else g["feed"]
    fov = max(g["nx"] * g["dx"], g["ny"] * (g["dy"] or g["dx"]))
    return synth.Geometry(synth.HELICAL, g["nx"], g["ny"], g["nz"], g["dx"], g["dy"] or g["dx"], g["dz"], g["cx"],
                          g["cy"], g["cz"], 570.0, 1040.0, g["V"], g["vpr"], g["start"], feed,
                          -feed * g["V"] / g["vpr"] / 2.0, g["R"], g["row_mm"] * 1040.0 / 570.0, g["K"],
                          synth.fan_pitch(fov / 2.0, 570.0, g["K"]), 0.25, g["row_offset"])


# columns enough to fill the GPU with two and with one group of views
LARGE = {
    "two_groups": _geo(nx=390, ny=261, nz=41, dx=0.98, K=150, V=9, vpr=9, pitch=3.0),
    "one_group": _geo(nx=512, ny=509, nz=49, dx=0.98, K=200, V=7, vpr=7, pitch=3.0),
    "slice_tilted_wide": _geo(nx=410, ny=397, nz=1, R=1, dx=0.9, K=150, V=11, vpr=11, feed=0.8),
    "slice_wide": _geo(nx=410, ny=397, nz=1, R=1, dx=0.9, K=150, V=11, vpr=11, feed=0.0),
}
GEOMETRIES = {
    # split over four view groups: deep and shallow slab class, exact and ragged slices
    "deep": _geo(nz=32),
    "deep_ragged": _geo(nx=37, ny=29, nz=17, K=101, V=53, vpr=61),
    "mid": _geo(nz=22, dz=1.5),
    "mid_ragged": _geo(nx=41, ny=33, nz=23, dz=1.5, R=11, K=83),
    # few rays per column, and more channels than one turn takes
    "coarse_fan": _geo(K=17),
    "fine_fan": _geo(nx=24, ny=20, dx=8.0, K=420, V=24, vpr=24),
    # many slices per row and per voxel edge: the rays of a row lie slices apart
    "straddling": _geo(nx=30, ny=30, nz=40, dx=8.0, dz=0.2, R=9, row_mm=2.0),
    "two_slices": _geo(nz=2, R=4),
    "one_row": _geo(nz=9, R=1, V=64, vpr=64),
    "one_column": _geo(nx=1, ny=1, nz=9, dx=60.0, K=33),
    "huge_voxels": _geo(nx=8, ny=7, nz=5, dx=60.0, dz=2.0, K=64),
    # one slice and one row: sixteen and eight warps per patch, in the plane of the
    # source and beside it
    "slice": _geo(nx=45, ny=34, nz=1, R=1, K=90, V=70, vpr=70, feed=0.0),
    "slice_few_views": _geo(nx=20, ny=19, nz=1, R=1, K=31, V=5, vpr=5, feed=0.0),
    "slice_tilted": _geo(nx=45, ny=34, nz=1, R=1, K=90, V=70, vpr=70, feed=0.6, row_offset=0.3),
    "off_axis": _geo(nx=33, ny=38, dy=5.1, cx=9.0, cy=-6.0, cz=1.3, row_offset=0.35, R=5, nz=19),
}


def _case(geo):
    return dataclasses.replace(synth.make_case("t3d"), geo=geo)


def _rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("name", sorted(GEOMETRIES))
def test_adjoint_matches_oracle(pkg, name):
    import oracle
    case = _case(GEOMETRIES[name])
    gpu = pkg.from_case(case)
    y = synth.random_rays(case.geo, 21).float()
    got = gpu.backproject(y.cuda()).cpu().numpy()
    ref = oracle.from_case(case).adjoint(y.double().numpy())
    assert _rel(got, ref) < 1e-5
    gpu.close()


@pytest.mark.parametrize("name", ["deep_ragged", "mid_ragged", "straddling", "two_slices", "one_row", "slice",
                                  "slice_tilted"])
def test_sums_and_gradient_match_adjoint_of_payload(pkg, name):
    import oracle
    case = _case(GEOMETRIES[name])
    gpu = pkg.from_case(case)
    gen = torch.Generator().manual_seed(3)
    geo = case.geo
    d = 1e5 * torch.rand((2, geo.n_views, geo.n_rows, geo.n_channels), generator=gen)
    c = 0.5 * torch.rand((geo.nz, geo.ny, geo.nx, 2), generator=gen)
    gpu.set_data(d.cuda())
    pay, _ = gpu.ray_terms(c.cuda())
    sums, _, _ = gpu.backprojected_sums(c.cuda())
    grad, _ = gpu.gradient(c.cuda())
    O = oracle.from_case(case)
    p = pay.cpu().double().numpy()
    for i in range(2):
        ref = O.adjoint(np.ascontiguousarray(p[..., 2 * i:2 * i + 2]))
        assert _rel(sums[..., 2 * i:2 * i + 2].cpu().numpy(), ref) < 1e-5
    assert torch.equal(grad, sums[..., 2:].contiguous())
    gpu.close()


@pytest.mark.parametrize("name", sorted(LARGE))
def test_adjoint_identity_of_large_plans(pkg, name):
    gpu = pkg.from_case(_case(LARGE[name]))
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.rand(gpu.img_shape, generator=gen, device="cuda")
    y = torch.rand(gpu.ray_shape + (2,), generator=gen, device="cuda")
    Ax, _ = gpu.forward(x)
    Aty = gpu.backproject(y)
    lhs = torch.sum(Ax.double() * y.double()).item()
    rhs = torch.sum(x.double() * Aty.double()).item()
    assert abs(lhs - rhs) <= 2e-6 * abs(lhs)
    gpu.close()
