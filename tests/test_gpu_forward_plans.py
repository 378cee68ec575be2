"""How many detector rows a thread of the forward projection takes follows the scan:
one where few views, a thin volume or steep rows leave nothing to share.  The scans
below have views enough for groups of 4 and 8 rows, with row counts around the group
sizes, cone beams off centre, thin and thick slices.

Line integrals against the oracle to the projections' bar (rel-L2 1e-5), and bit for
bit those of the same scan cut to its first eight views, which runs one row per
thread with the same arithmetic."""
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


def _geo(R, nz, dz, V, K=70, nx=36, ny=32, dx=4.0, row_offset=0.0, cz=0.0, vpr=None):
    feed = 0.8 * R * 0.75
    return synth.Geometry(synth.HELICAL, nx, ny, nz, dx, dx, dz, 0.0, 0.0, cz, 570.0, 1040.0, V, vpr or V, 0.3, feed,
                          -feed / 2.0, R, 0.75 * 1040.0 / 570.0, K, synth.fan_pitch(nx * dx / 2.0, 570.0, K), 0.25,
                          row_offset)


GROUPS = {
    "rows2": (4, _geo(2, 6, 0.75, 2320)), "rows3": (4, _geo(3, 8, 0.75, 2320)), "rows4": (4, _geo(4, 12, 0.75, 2320)),
    "rows5": (8, _geo(5, 17, 0.75, 1560)), "rows8": (8, _geo(8, 30, 0.75, 1560)),
    "rows9": (8, _geo(9, 33, 0.75, 800, K=65)), "rows15": (8, _geo(15, 61, 0.75, 800)),
    "rows16_thick_slices": (8, _geo(16, 20, 1.5, 408)), "rows16_steep": (8, _geo(16, 60, 0.55, 1080)),
    "rows33": (8, _geo(33, 80, 1.0, 240)), "thin_volume": (4, _geo(16, 12, 0.75, 600)),
    "thin_volume_rows11": (4, _geo(11, 9, 0.75, 800)), "off_centre": (8, _geo(16, 40, 1.0, 600, row_offset=0.35, cz=6.0)),
    "far_off": (8, _geo(16, 40, 1.0, 600, row_offset=-11.0, cz=-9.0)),
}


def _case(geo):
    return dataclasses.replace(synth.make_case("t3d"), geo=geo)


@pytest.mark.parametrize("name", sorted(GROUPS))
def test_groups_of_rows(pkg, name):
    import oracle
    rows, geo = GROUPS[name]
    case, cut = _case(geo), _case(geo.replace(n_views=8))
    gpu, few = pkg.from_case(case), pkg.from_case(cut)
    assert gpu.kernel_plan()["fwd_rows"] == rows and few.kernel_plan()["fwd_rows"] == 1
    c = synth.random_image(geo, 3).float()
    l, g = gpu.forward(c.cuda(), want_g=True)
    ref = oracle.from_case(case).forward(c.double().numpy())
    got = l.cpu().double().numpy()
    assert np.linalg.norm(got - ref) < 1e-5 * np.linalg.norm(ref)
    assert np.array_equal(got[ref.max(-1) == 0], ref[ref.max(-1) == 0])  # rays beside the volume: exactly zero
    assert torch.equal(l[:8], few.forward(c.cuda())[0])
    # the objective from groups of rows: that of the batched plan, one row per thread (1e-12, two orders of FP64 sums)
    d = 1e5 * torch.rand((2,) + gpu.ray_shape, generator=torch.Generator().manual_seed(1)).cuda()
    gpu.set_data(d)
    batch = pkg.DeamBatch([gpu], autotune=False)
    H = batch.iterate([c.cuda().contiguous()], 1)
    np.testing.assert_allclose(H[0, 0], gpu.objective(c.cuda()), rtol=1e-12)
    batch.close()
    gpu.close()
    few.close()


@pytest.mark.parametrize("rows,kw", [
    (1, dict(R=16, nz=32, dz=0.75, V=36)), (1, dict(R=16, nz=32, dz=0.75, V=150)), (4, dict(R=16, nz=32, dz=0.75, V=180)),
    (8, dict(R=16, nz=32, dz=0.75, V=360)), (1, dict(R=16, nz=32, dz=1.5, V=60)), (8, dict(R=16, nz=32, dz=1.5, V=120)),
    (1, dict(R=16, nz=9, dz=0.75, V=720)), (4, dict(R=16, nz=10, dz=0.75, V=720)),
    (1, dict(R=16, nz=60, dz=0.4, V=720)), (8, dict(R=16, nz=60, dz=0.55, V=720)),
    (1, dict(R=1, nz=16, dz=0.75, V=720))])
def test_rows_follow_the_scan(pkg, rows, kw):
    gpu = pkg.from_case(_case(_geo(K=300, nx=64, ny=64, **kw)))
    assert gpu.kernel_plan()["fwd_rows"] == rows
    gpu.close()
