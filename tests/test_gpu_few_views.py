"""The backprojection of scans with few views: as many warps share the views of a
column as have views to take, and views whose rays lie slices apart are taken one at
a time.  Every slab depth, columns that fill the GPU and columns that do not, view
counts around the eights that a warp takes.

Against the oracle's adjoint to rel-L2 2 N 2^-23 on planes of N voxels (FP32 in-plane
positions up to N are off by 2^-23 N at most, which moves that share of a sample's
weight, one half on average, to the next voxel), and never tighter than the
backprojection's bar of 1e-5."""
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


def _check(pkg, plan, nx, nz, V, R=16, dz=0.75, dx=0.98, K=None, vpr=None, feed=None):
    import oracle
    K = K or (5 * nx) // 3
    vpr = vpr or 96
    feed = min(9.6, 0.2 * dz * vpr) if feed is None else feed  # neighbouring views a fraction of a slice apart
    geo = synth.Geometry(synth.HELICAL, nx, nx - 3, nz, dx, dx, dz, 0.0, 0.0, 0.0, 570.0, 1040.0, V, vpr, 0.3, feed,
                         -feed * V / vpr / 2.0, R, 0.75 * 1040.0 / 570.0, K,
                         synth.fan_pitch(nx * dx / 2.0, 570.0, K), 0.25, 0.0)
    case = dataclasses.replace(synth.make_case("t3d"), geo=geo)
    gpu = pkg.from_case(case)
    got = gpu.kernel_plan()
    slab, groups, views = plan
    assert got["bwd_slab"] == slab and got["bwd_views"] == views
    assert groups is None or got["bwd_groups"] == groups
    y = synth.random_rays(geo, 21).float()
    img = gpu.backproject(y.cuda()).cpu().double().numpy()
    ref = oracle.from_case(case).adjoint(y.double().numpy())
    assert np.linalg.norm(img - ref) < max(1e-5, 2.0 * nx * 2.0**-23) * np.linalg.norm(ref)
    gpu.close()


@pytest.mark.parametrize("V,groups", [(8, 1), (9, 2), (16, 2), (17, 4), (40, 4)])
@pytest.mark.parametrize("slab,nz,dz,R", [(16, 12, 0.75, 16), (11, 12, 1.5, 16), (2, 2, 0.75, 4)])
def test_columns_that_do_not_fill_the_gpu(pkg, slab, nz, dz, R, V, groups):
    _check(pkg, (slab, groups, 2), 40, nz, V, R=R, dz=dz, dx=4.0)


@pytest.mark.parametrize("slab,nz,dz,V,groups", [
    (16, 32, 0.75, 8, 1), (16, 32, 0.75, 24, 1), (16, 32, 0.75, 32, 2), (16, 32, 0.75, 60, 4),
    (11, 32, 1.5, 24, 1), (11, 32, 1.5, 33, 2), (11, 32, 1.5, 57, 4),
    (2, 2, 0.75, 8, 1), (2, 2, 0.75, 16, 2), (2, 2, 0.75, 56, 2), (2, 2, 0.75, 64, 4)])
def test_columns_that_fill_the_gpu(pkg, slab, nz, dz, V, groups):
    _check(pkg, (slab, groups, 2), 256, nz, V, dz=dz)


@pytest.mark.parametrize("V,vpr", [(1, 1), (2, 2), (3, 3), (7, 7), (20, 7), (33, 5), (16, 2)])
@pytest.mark.parametrize("slab,nz,dz,R", [(16, 20, 0.75, 16), (11, 14, 1.5, 5), (2, 2, 0.75, 4), (11, 9, 0.75, 1)])
def test_views_far_apart_in_angle(pkg, slab, nz, dz, R, V, vpr):
    # over several rotations some views pass a slab by
    _check(pkg, (slab, 1 if V <= 8 else None, 1), 40, nz, V, R=R, dz=dz, dx=4.0, vpr=vpr)


@pytest.mark.parametrize("slices", [1.0, 2.3, -1.5])
@pytest.mark.parametrize("slab,nz,dz,R", [(16, 24, 0.75, 9), (11, 24, 1.5, 5), (11, 24, 0.75, 1)])
def test_views_far_apart_in_height(pkg, slab, nz, dz, R, slices):
    # (views enough to reach every slab; how many reach one, and so its warps, depends on the step)
    _check(pkg, (slab, None, 1), 40, nz, 23, R=R, dz=dz, dx=4.0, vpr=60, feed=slices * dz * 60)
