"""The backprojection of detectors whose channels are coarse against the voxels: a
turn takes one ray of a view or two.  From rays that most columns never meet up to the
change to four rays per turn, every slab depth and number of warps per column.

Against the oracle's adjoint to rel-L2 2 N 2^-23 on planes of N voxels (FP32 in-plane
positions up to N are off by 2^-23 N at most, which moves that share of a sample's
weight, one half on average, to the next voxel), and never tighter than the
backprojection's bar of 1e-5; the gradient equals the fused sums' second pair."""
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


def _case(nx, nz, V, R, dz, dx, K):
    geo = synth.Geometry(synth.HELICAL, nx, nx - 3, nz, dx, dx, dz, 0.0, 0.0, 0.0, 570.0, 1040.0, V, 96, 0.3,
                         0.2 * dz * 96, -0.1 * dz * V, R, 0.75 * 1040.0 / 570.0, K,
                         synth.fan_pitch(nx * dx / 2.0, 570.0, K), 0.25, 0.0)
    return dataclasses.replace(synth.make_case("t3d"), geo=geo)


@pytest.mark.parametrize("K,rays", [(2, 1), (7, 1), (15, 1), (17, 2), (40, 2), (43, 2), (50, 4)])
@pytest.mark.parametrize("nz,dz,R", [(18, 0.75, 16), (13, 1.5, 11), (2, 0.75, 4), (9, 0.75, 1)])
def test_rays_per_turn(pkg, K, rays, nz, dz, R):
    import oracle
    case = _case(40, nz, 50, R, dz, 4.0, K)
    gpu = pkg.from_case(case)
    assert gpu.kernel_plan()["bwd_rays"] == rays
    geo = case.geo
    y = synth.random_rays(geo, 21).float()
    img = gpu.backproject(y.cuda()).cpu().double().numpy()
    ref = oracle.from_case(case).adjoint(y.double().numpy())
    assert np.linalg.norm(img - ref) < 1e-5 * np.linalg.norm(ref)
    gen = torch.Generator().manual_seed(3)
    gpu.set_data((1e5 * torch.rand((2,) + gpu.ray_shape, generator=gen)).cuda())
    c = (0.5 * torch.rand(gpu.img_shape, generator=gen)).cuda()
    sums, _, _ = gpu.backprojected_sums(c)
    grad, _ = gpu.gradient(c)
    assert torch.equal(grad, sums[..., 2:].contiguous())
    gpu.close()


@pytest.mark.parametrize("K,rays", [(120, 1), (250, 2)])
@pytest.mark.parametrize("groups,nx,nz,dz", [(1, 512, 49, 0.75), (2, 390, 57, 0.75), (1, 512, 31, 1.5), (2, 390, 41, 1.5)])
def test_large_volumes(pkg, groups, nx, nz, dz, K, rays):
    import oracle
    case = _case(nx, nz, 300, 9, dz, 0.98, K)
    gpu = pkg.from_case(case)
    plan = gpu.kernel_plan()
    assert (plan["bwd_rays"], plan["bwd_groups"]) == (rays, groups)
    y = synth.random_rays(case.geo, 21).float()
    img = gpu.backproject(y.cuda()).cpu().double().numpy()
    ref = oracle.from_case(case).adjoint(y.double().numpy())
    assert np.linalg.norm(img - ref) < 2.0 * nx * 2.0**-23 * np.linalg.norm(ref)
    gpu.close()
