"""The ramp filter and the FBP sums at the edges of their work split: channel
counts around the four outputs of a thread and both parities, rows around the
rows of a block, one to three slices for threads that take two, the longest row
(more than 48 KB of shared memory for two spectra).

Against the FP64 oracle to the FBP's bar (relative L2 1e-4, FP32 fan angles times
the filtered sinogram's channel-to-channel variation); one spectrum against two to
1e-6.  The fan covers the image's corners, so that no voxel lies on the edge of
the detector, where FP32 and FP64 may differ on whether a view sees it."""
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


@pytest.mark.parametrize("K,R,nz,V", [(3, 2, 1, 30), (4, 1, 1, 30), (5, 3, 2, 31), (8, 1, 1, 30), (9, 4, 3, 30),
                                      (10, 2, 5, 30), (63, 5, 3, 30), (64, 1, 1, 30), (65, 3, 2, 31), (66, 2, 1, 30),
                                      (383, 3, 3, 13), (512, 1, 1, 13), (767, 1, 1, 13), (3071, 2, 2, 12),
                                      (3072, 1, 1, 12)])
def test_fbp_edges(pkg, K, R, nz, V):
    import oracle
    nx, ny, dx = 36, 32, 4.0
    feed = 0.8 * R * 0.75 if R > 1 else 0.0
    kind = synth.HELICAL if R > 1 else synth.FAN2D
    pitch = synth.fan_pitch(0.75 * nx * dx, 570.0, K) * (K + 1) / (K - 1)
    geo = synth.Geometry(kind, nx, ny, nz, dx, dx, 0.75, 0.0, 0.0, 0.0, 570.0, 1040.0, V, V, 0.3, feed, -feed / 2.0, R,
                         0.75 * 1040.0 / 570.0, K, pitch, 0.25 if K > 3 else 0.0, 0.0)
    case = dataclasses.replace(synth.make_case("t3d"), geo=geo)
    d, _ = synth.measure(case, seed=1, noiseless=True)
    g = pkg.from_case(case)
    g.set_data(d.cuda())
    O = oracle.from_case(case)
    p = torch.from_numpy(O.log_sinogram(d.double().numpy(), 1.0) + 0.3).float().contiguous()
    img = g.fbp(p.cuda()).cpu().double().numpy()
    for j in range(2):
        ref = O.fbp(p[j].double().numpy())
        assert np.linalg.norm(img[j] - ref) < 1e-4 * np.linalg.norm(ref)
        one = g.fbp(p[j].contiguous().cuda()).cpu().double().numpy()
        assert np.linalg.norm(one - img[j]) < 1e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("kind", ["none", "ray", "per_spectrum", "everywhere"])
@pytest.mark.parametrize("R,nz", [(1, 1), (3, 4), (9, 40)])
def test_mar_init_equals_its_steps(pkg, kind, R, nz):
    # the initialisation projects the prior along the rays that completion reads:
    # bit for bit the images of the same steps with all rays projected
    nx, ny, dx, K, V = 36, 32, 4.0, 70, 20
    feed = 0.8 * R * 0.75 if R > 1 else 0.0
    geo = synth.Geometry(synth.HELICAL if R > 1 else synth.FAN2D, nx, ny, nz, dx, dx, 0.75, 0.0, 0.0, 0.0, 570.0, 1040.0,
                         V, V, 0.3, feed, -feed / 2.0, R, 0.75 * 1040.0 / 570.0, K,
                         synth.fan_pitch(0.5 * nx * dx, 570.0, K), 0.25, 0.0)
    case = dataclasses.replace(synth.make_case("t3d"), geo=geo)
    d, _ = synth.measure(case, seed=1)
    gen = torch.Generator().manual_seed(7)
    g = pkg.from_case(case)
    g.set_data(d.cuda())
    shape = (V, R, K)
    if kind == "per_spectrum":
        g.set_metal_mask((torch.rand((2,) + shape, generator=gen) < 0.1).to(torch.uint8).cuda(), "per_spectrum")
    elif kind != "none":
        m = torch.rand(shape, generator=gen) < (0.03 if kind == "ray" else 2.0)
        m[::3, :, 0], m[1::3, :, K - 1], m[2, R // 2] = True, True, True
        g.set_metal_mask(m.to(torch.uint8).cuda(), "ray")
    prior = (0.03 * torch.rand((nz, ny, nx), generator=gen)).cuda()
    _, _, mu = g.mar_init([1.0, 0.1, 0.9, 0.4], 0.005, 0.026, 0.0195, prior=prior)
    p = g.log_sinogram()
    l, _ = g.forward(torch.stack([prior, torch.zeros_like(prior)], -1).contiguous())
    line = l[..., 0].contiguous()
    t = torch.stack([g.complete_trace(p[j].contiguous(), j, prior_proj=line) for j in range(2)])
    ref = g.fbp(t.contiguous())
    assert torch.equal(mu.reshape(ref.shape), ref)
