"""FBP with one and with two slices per thread (two from 16 warps per SM up), on
detectors of one row and of several, with odd and even slices; few rows spread over
the GPU and many packed into blocks.  Against the FP64 oracle to the FBP's bar
(relative L2 1e-4); the middle slice of a volume is the same bit for bit as that slice
alone, whichever plan each runs."""
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


def _scan(pkg, nx, nz, R, K, V):
    feed = 0.8 * R * 0.75 if R > 1 else 0.0
    pitch = synth.fan_pitch(0.75 * nx * 0.98, 570.0, K) * (K + 1) / (K - 1)
    geo = synth.Geometry(synth.HELICAL, nx, nx, nz, 0.98, 0.98, 0.75, 0.0, 0.0, 0.0, 570.0, 1040.0, V, V, 0.3, feed,
                         -feed / 2.0, R, 0.75 * 1040.0 / 570.0, K, pitch, 0.25, 0.0)
    case = dataclasses.replace(synth.make_case("t3d"), geo=geo)
    s = pkg.from_case(case)
    s.set_data(torch.ones((2, V, R, K)).cuda())
    return case, s


@pytest.mark.parametrize("R", [1, 4])
@pytest.mark.parametrize("nx,nz", [(160, 3), (160, 9), (240, 11), (240, 12)])  # below and above 2432 warps
def test_slices_per_thread(pkg, nx, nz, R):
    import oracle
    K, V = 200, 24
    case, s = _scan(pkg, nx, nz, R, K, V)
    p = (0.3 + torch.rand((2, V, R, K), generator=torch.Generator().manual_seed(2))).cuda()
    img = s.fbp(p)
    O = oracle.from_case(case)
    for j in range(2):
        ref = O.fbp(p[j].cpu().double().numpy())
        assert np.linalg.norm(img[j].cpu().double().numpy() - ref) < 1e-4 * np.linalg.norm(ref)
    # the middle slice alone (an odd volume's is at the same height to the bit)
    if nz % 2:
        _, one = _scan(pkg, nx, 1, R, K, V)
        assert torch.equal(one.fbp(p)[:, 0], img[:, nz // 2])
        one.close()
    s.close()


@pytest.mark.parametrize("K,V", [(9, 1500), (9, 230), (64, 1500)])
def test_rows_per_block(pkg, K, V):
    # rows enough to fill blocks (as many as 64 to a block at 9 channels) and some that
    # are spread over the GPU first
    import oracle
    R, nx = 8, 24
    case, s = _scan(pkg, nx, 3, R, K, V)
    p = (0.3 + torch.rand((2, V, R, K), generator=torch.Generator().manual_seed(2))).cuda()
    img = s.fbp(p)
    O = oracle.from_case(case)
    for j in range(2):
        ref = O.fbp(p[j].cpu().double().numpy())
        assert np.linalg.norm(img[j].cpu().double().numpy() - ref) < 1e-4 * np.linalg.norm(ref)
    s.close()
