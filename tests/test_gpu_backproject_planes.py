"""The backprojection of views whose rays lie in a slice but for the rounding of
their height: the forward kernel gives such a sample to the slice with all of its
weight, whichever side of it the rounding leaves the height on, and so must the
gather, next to views that are well above or below.

The detector's middle row is horizontal, so that all its samples are as high as the
source.  Against the oracle's adjoint to the backprojection's bar (rel-L2 1e-5)."""
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


# nz, dz, rows: slabs of 2, 11 (one row, thick slices) and 16 slices
SLABS = [(2, 0.75, 3), (7, 0.75, 1), (12, 1.5, 3), (21, 0.75, 3)]


@pytest.mark.parametrize("nz,dz,R", SLABS)
@pytest.mark.parametrize("view", [0, 1, 6])
@pytest.mark.parametrize("above", [-2e-8, -1e-9, 0.0, 1e-9])
def test_view_at_the_height_of_a_slice(pkg, nz, dz, R, view, above):
    import oracle
    nx, ny, dx, K, V = 24, 20, 4.0, 40, 16
    step = 0.05 * dz  # of the source per view
    # view `view` is `above` slices above the lowest one
    start = -(nz - 1) / 2.0 * dz + above * dz - view * step
    geo = synth.Geometry(synth.HELICAL, nx, ny, nz, dx, dx, dz, 0.0, 0.0, 0.0, 570.0, 1040.0, V, V, 0.3, step * V, start,
                         R, 0.75 * 1040.0 / 570.0, K, synth.fan_pitch(nx * dx / 2.0, 570.0, K), 0.25, 0.0)
    case = dataclasses.replace(synth.make_case("t3d"), geo=geo)
    gpu = pkg.from_case(case)
    y = torch.zeros(gpu.ray_shape + (2,))
    y[:, R // 2] = synth.random_rays(geo, 21).float()[:, R // 2]
    got = gpu.backproject(y.cuda()).cpu().double().numpy()
    ref = oracle.from_case(case).adjoint(y.double().numpy())
    assert np.linalg.norm(got - ref) < 1e-5 * np.linalg.norm(ref)
    gpu.close()
