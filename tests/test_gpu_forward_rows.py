"""The forward projection with several detector rows per thread (1, 4 or 8, by the
detector and the height of the volume): row counts around the group sizes, rows
rising by a fraction of a slice and by several, thin volumes that most rows leave,
cone beams off centre.

Line integrals against the oracle to the projections' bar (rel-L2 1e-5); the
objective against the batched persistent plan, which projects one row per thread
with the same arithmetic, to the bar of two FP64 summation orders (1e-12)."""
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


def _geo(R, nz, dz, row_mm=0.75, K=70, V=40, nx=36, ny=32, row_offset=0.0, cz=0.0, pitch=0.8):
    feed = pitch * R * row_mm
    dx = 4.0
    return synth.Geometry(synth.HELICAL, nx, ny, nz, dx, dx, dz, 0.0, 0.0, cz, 570.0, 1040.0, V, V, 0.3, feed,
                          -feed / 2.0, R, row_mm * 1040.0 / 570.0, K, synth.fan_pitch(nx * dx / 2.0, 570.0, K), 0.25,
                          row_offset)


GEOMETRIES = {
    "rows2": _geo(2, 6, 0.75), "rows3": _geo(3, 8, 0.75), "rows4": _geo(4, 12, 0.75), "rows5": _geo(5, 17, 0.75),
    "rows8": _geo(8, 30, 0.75), "rows9": _geo(9, 33, 0.75, K=65), "rows15": _geo(15, 61, 0.75, V=17),
    "rows16_thick_slices": _geo(16, 20, 1.5), "rows16_thin_slices": _geo(16, 200, 0.2, V=19),
    "rows33": _geo(33, 80, 1.0, V=13),
    "thin_volume": _geo(16, 5, 0.75), "thin_volume_steep": _geo(16, 9, 0.2), "one_slice": _geo(6, 1, 0.75),
    "off_centre": _geo(16, 40, 1.0, row_offset=0.35, cz=6.0), "far_off": _geo(16, 40, 1.0, row_offset=-11.0, cz=-9.0),
}


def _case(geo):
    return dataclasses.replace(synth.make_case("t3d"), geo=geo)


@pytest.mark.parametrize("name", sorted(GEOMETRIES))
def test_line_integrals_match_oracle(pkg, name):
    import oracle
    case = _case(GEOMETRIES[name])
    gpu = pkg.from_case(case)
    c = synth.random_image(case.geo, 3).float()
    l, g = gpu.forward(c.cuda(), want_g=True)
    O = oracle.from_case(case)
    ref = O.forward(c.double().numpy())
    got = l.cpu().double().numpy()
    assert np.linalg.norm(got - ref) < 1e-5 * np.linalg.norm(ref)
    assert np.array_equal(got[ref.max(-1) == 0], ref[ref.max(-1) == 0])   # rays beside the volume: exactly zero
    l2, _ = gpu.forward(c.cuda())
    assert torch.equal(l, l2)
    gpu.close()


def test_objective_equals_one_row_per_thread(pkg):
    scans, images = [], []
    gen = torch.Generator().manual_seed(1)
    for name in ("rows3", "rows9", "rows15", "thin_volume", "rows16_thin_slices"):
        case = _case(GEOMETRIES[name])
        geo = case.geo
        s = pkg.from_case(case)
        s.set_data((1e5 * torch.rand((2, geo.n_views, geo.n_rows, geo.n_channels), generator=gen)).cuda())
        scans.append(s)
        images.append((0.3 * torch.rand((geo.nz, geo.ny, geo.nx, 2), generator=gen)).cuda())
    alone = [s.objective(c) for s, c in zip(scans, images)]
    batch = pkg.DeamBatch(scans, autotune=False)
    H = batch.iterate([c.clone() for c in images], 1)
    np.testing.assert_allclose(H[:, 0], alone, rtol=1e-12)
    batch.close()


@pytest.mark.parametrize("name", ["narrow", "wide", "one_row_helical"])
def test_objective_of_single_rows(pkg, name):
    # one row per thread: blocks of four and of eight warps, whose last one adds up
    # the objective; against the batched plan (1e-12), and the same on every call
    K, V, nz, nx = {"narrow": (31, 9, 1, 20), "wide": (640, 260, 1, 40), "one_row_helical": (70, 333, 7, 24)}[name]
    geo = synth.Geometry(synth.HELICAL, nx, nx, nz, 4.0, 4.0, 0.75, 0.0, 0.0, 0.0, 570.0, 1040.0, V, V, 0.3,
                         0.6 if nz > 1 else 0.0, -0.3 if nz > 1 else 0.0, 1, 0.75 * 1040.0 / 570.0, K,
                         synth.fan_pitch(nx * 2.0, 570.0, K), 0.25, 0.0)
    s = pkg.from_case(_case(geo))
    gen = torch.Generator().manual_seed(1)
    s.set_data((1e5 * torch.rand((2, V, 1, K), generator=gen)).cuda())
    c = (0.3 * torch.rand((nz, nx, nx, 2), generator=gen)).cuda()
    F = [s.objective(c) for _ in range(3)]
    assert F[0] == F[1] == F[2]
    H = s.iterate(c.clone(), 3)
    info = s.info()
    batch = pkg.DeamBatch([s], autotune=False)
    B = batch.iterate([c.clone()], 3)
    np.testing.assert_allclose(B[0, 0], F[0], rtol=1e-12)
    np.testing.assert_allclose(H[0], F[0], rtol=1e-12)
    np.testing.assert_allclose(H, B[0], rtol=1e-7)
    assert np.array_equal(s.iterate(c.clone(), 3), H) and s.info() == info   # skipped voxels counted anew
    batch.close()
