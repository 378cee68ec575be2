"""The plans of the backprojection (Deam.kernel_plan says which) at their usual four
rays per turn: every slab depth with one, two and four warps per column, two views a
turn and one, and single slices
with 2 x 2 columns per thread around the edges of their 16 x 8 patches, few and many
rays per column, views around the eights that a warp takes, rays in the slice and
beside it.

Voxel by voxel against the oracle's adjoint to rel-L2 2 N 2^-23 for planes of N
voxels: FP32 in-plane positions up to N are off by 2^-23 N at most (the intercept and
the slope's product, half a unit in the last place of N each), which moves that share
of a sample's weight, one half on average, to the next voxel.  And by the adjoint
identity to the bar that the other identities have."""
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


def _case(nx, ny, nz, R, K, V, dz=0.75, dx=0.98, feed=None):
    feed = (1.2 * R if R > 1 else 0.0) if feed is None else feed
    geo = synth.Geometry(synth.HELICAL, nx, ny, nz, dx, dx, dz, 0.0, 0.0, 0.0, 570.0, 1040.0, V, V, 0.3, feed,
                         -feed / 2.0, R, 0.75 * 1040.0 / 570.0, K,
                         synth.fan_pitch(max(nx, ny) * dx / 2.0, 570.0, K), 0.25, 0.0)
    return dataclasses.replace(synth.make_case("t3d"), geo=geo)


def _check(pkg, case, slab, groups, views, rays):
    import oracle
    gpu = pkg.from_case(case)
    plan = gpu.kernel_plan()
    assert (plan["bwd_slab"], plan["bwd_groups"], plan["bwd_views"], plan["bwd_rays"]) == (slab, groups, views, rays)
    geo = case.geo
    y = synth.random_rays(geo, 21).float()
    got = gpu.backproject(y.cuda())
    ref = oracle.from_case(case).adjoint(y.double().numpy())
    off = np.linalg.norm(got.cpu().double().numpy() - ref)
    assert off < 2.0 * max(geo.nx, geo.ny) * 2.0**-23 * np.linalg.norm(ref)
    x = torch.rand(gpu.img_shape, generator=torch.Generator().manual_seed(5)).cuda()
    lines, _ = gpu.forward(x)
    lhs = torch.sum(lines.double() * y.cuda().double()).item()
    rhs = torch.sum(x.double() * got.double()).item()
    assert abs(lhs - rhs) <= 2e-6 * abs(lhs)
    gpu.close()


@pytest.mark.parametrize("V,views", [(200, 2), (70, 1)])  # the source 0.2-0.3 and 0.4-0.8 slices further per view
@pytest.mark.parametrize("slab,groups,nx,ny,nz,dz,K", [
    (16, 2, 390, 261, 57, 0.75, 480), (16, 1, 512, 509, 49, 0.75, 620),
    (11, 2, 390, 261, 41, 1.5, 480), (11, 1, 512, 509, 31, 1.5, 620)])
def test_large_slabs(pkg, slab, groups, nx, ny, nz, dz, K, V, views):
    # the source travels the height of the volume, 25 views or more past each slab
    _check(pkg, _case(nx, ny, nz, 9, K, V, dz=dz, feed=nz * dz), slab, groups, views, 4)


@pytest.mark.parametrize("feed", [0.0, 0.7])
@pytest.mark.parametrize("nx,ny,K,V", [(304, 264, 300, 8), (305, 263, 100, 7), (303, 265, 1300, 9), (289, 271, 420, 19),
                                       (513, 153, 700, 16)])
def test_slices_of_many_patches(pkg, nx, ny, K, V, feed):
    _check(pkg, _case(nx, ny, 1, 1, K, V, feed=feed), 1, 8, 1, 1)


@pytest.mark.parametrize("slab,nz,dz,R", [(16, 30, 0.75, 16), (11, 17, 1.5, 16), (2, 2, 0.75, 4)])
@pytest.mark.parametrize("V", [97, 250])
def test_four_warps_per_column(pkg, slab, nz, dz, R, V):
    _check(pkg, _case(61, 58, nz, R, 90, V, dz=dz, dx=2.5, feed=min(nz * dz, 0.3 * dz * V)), slab, 4, 2, 4)
