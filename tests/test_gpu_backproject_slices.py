"""The backprojection of single slices, whose threads take 2 x 2 columns: images
around the 16 x 8 columns of a block, few and many rays per column, views around the
eights that a warp takes, both numbers of warps, rays in the slice and beside it.

Against the oracle's adjoint to the backprojection's bar (rel-L2 1e-5), and on images
of many blocks by the adjoint identity (2e-6).  Infinities and NaN in a ray reach the
voxels that the ray taps and no other, bit for bit."""
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


def _case(nx, ny, K, V, feed=0.0, dx=4.0):
    fov = max(nx, ny) * dx
    geo = synth.Geometry(synth.HELICAL, nx, ny, 1, dx, dx, 0.75, 0.0, 0.0, 0.0, 570.0, 1040.0, V, V, 0.3, feed,
                         -feed / 2.0, 1, 0.75 * 1040.0 / 570.0, K, synth.fan_pitch(fov / 2.0, 570.0, K), 0.25, 0.0)
    return dataclasses.replace(synth.make_case("t3d"), geo=geo)


@pytest.mark.parametrize("feed", [0.0, 0.7])
@pytest.mark.parametrize("nx,ny,K,V", [(2, 2, 9, 8), (15, 7, 30, 7), (16, 8, 30, 8), (17, 9, 31, 9), (33, 5, 80, 130),
                                       (3, 40, 90, 17), (64, 64, 33, 40), (40, 40, 400, 24)])
def test_adjoint_matches_oracle(pkg, nx, ny, K, V, feed):
    import oracle
    case = _case(nx, ny, K, V, feed)
    gpu = pkg.from_case(case)
    y = synth.random_rays(case.geo, 21).float()
    got = gpu.backproject(y.cuda()).cpu().double().numpy()
    ref = oracle.from_case(case).adjoint(y.double().numpy())
    assert np.linalg.norm(got - ref) < 1e-5 * np.linalg.norm(ref)
    gpu.close()


@pytest.mark.parametrize("feed", [0.0, 0.7])
@pytest.mark.parametrize("nx,ny", [(305, 263), (300, 255)])
def test_adjoint_identity_of_many_blocks(pkg, nx, ny, feed):
    gpu = pkg.from_case(_case(nx, ny, 300, 19, feed, dx=0.98))
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.rand(gpu.img_shape, generator=gen, device="cuda")
    y = torch.rand(gpu.ray_shape + (2,), generator=gen, device="cuda")
    Ax, _ = gpu.forward(x)
    Aty = gpu.backproject(y)
    lhs = torch.sum(Ax.double() * y.double()).item()
    rhs = torch.sum(x.double() * Aty.double()).item()
    assert abs(lhs - rhs) <= 2e-6 * abs(lhs)
    gpu.close()


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("nx,ny,K,V,feed", [(45, 34, 90, 70, 0.0), (45, 34, 90, 70, 0.7), (305, 263, 300, 9, 0.0)])
def test_nonfinite_rays_stay_on_their_voxels(pkg, nx, ny, K, V, feed, value):
    gpu = pkg.from_case(_case(nx, ny, K, V, feed, dx=4.0 if nx < 100 else 0.98))
    y = torch.rand(gpu.ray_shape + (2,), generator=torch.Generator().manual_seed(2)).cuda()
    at = [(0, 0, K // 2), (V // 2, 0, K // 3)]
    one = torch.zeros_like(y)
    for i in at:
        y[i] = 0.0
        one[i] = 1.0
    taps = gpu.backproject(one) != 0
    ref = gpu.backproject(y)
    for i in at:
        y[i] = value
    got = gpu.backproject(y)
    assert taps.any() and not taps.all()
    assert torch.equal(torch.isfinite(got), ~taps)
    assert torch.equal(got[~taps], ref[~taps])
    gpu.close()
