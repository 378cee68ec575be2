"""The objective of a scan alone and in a batch that runs every scan's own kernels is
the same to the bit, whichever kernel adds it up: slices and slabs of one row per
thread (whose forward kernel's last block does), from one ray tile to thousands, in
blocks of four and of eight warps, and slabs of rows in groups."""
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
    import paper_2202_00116_gb300 as p
    return p


SCANS = [  # nx, nz, R, K, V: ray tiles 1, 4, 33, 180, 720, 4440, ...
    (12, 1, 1, 20, 3), (20, 1, 1, 31, 15), (24, 1, 1, 90, 85), (48, 1, 1, 120, 180), (64, 1, 1, 256, 360),
    (64, 1, 1, 640, 1777), (40, 5, 3, 70, 50), (40, 12, 16, 64, 60), (32, 3, 5, 100, 2000), (40, 20, 16, 70, 900)]


@pytest.mark.parametrize("precision", ["mixed", "fp32"])
def test_alone_and_in_a_batch(pkg, precision):
    scans, images = [], []
    for i, (nx, nz, R, K, V) in enumerate(SCANS):
        feed = 0.6 * R if R > 1 else 0.0
        geo = synth.Geometry(synth.HELICAL, nx, nx, nz, 4.0, 4.0, 0.75, 0.0, 0.0, 0.0, 570.0, 1040.0, V, V, 0.3, feed,
                             -feed / 2.0, R, 0.75 * 1040.0 / 570.0, K, synth.fan_pitch(nx * 2.0, 570.0, K), 0.25, 0.0)
        s = pkg.from_case(dataclasses.replace(synth.make_case("t3d"), geo=geo), precision=precision)
        gen = torch.Generator().manual_seed(i)
        # counts over five decades: terms that do not add up exactly in 53 bits
        s.set_data((10.0 ** (5.0 * torch.rand((2,) + s.ray_shape, generator=gen))).cuda())
        scans.append(s)
        images.append((0.1 * torch.rand(s.img_shape, generator=gen)).cuda())
    alone = [c.clone() for c in images]
    H = [s.iterate(c, 3) for s, c in zip(scans, alone)]
    together = [c.clone() for c in images]
    batch = pkg.DeamBatch(scans, plan="per_scan")
    B = batch.iterate(together, 3)
    for h, b, x, y, s, c in zip(H, B, alone, together, scans, images):
        np.testing.assert_array_equal(h, b)
        assert torch.equal(x, y)
        assert s.objective(c) == h[0]
    batch.close()


def test_many_tiles_and_data_sets(pkg):
    # 4440 partial sums: another order of them gave another last digit for one data set
    # in five
    K, V = 640, 1777
    geo = synth.Geometry(synth.FAN2D, 64, 64, 1, 4.0, 4.0, 0.75, 0.0, 0.0, 0.0, 570.0, 1040.0, V, V, 0.3, 0.0, 0.0, 1,
                         0.75 * 1040.0 / 570.0, K, synth.fan_pitch(128.0, 570.0, K), 0.25, 0.0)
    s = pkg.from_case(dataclasses.replace(synth.make_case("t3d"), geo=geo))
    for seed in range(20):
        gen = torch.Generator().manual_seed(seed)
        s.set_data((10.0 ** (5.0 * torch.rand((2,) + s.ray_shape, generator=gen))).cuda())
        c = (0.1 * torch.rand(s.img_shape, generator=gen)).cuda()
        batch = pkg.DeamBatch([s], plan="per_scan")
        np.testing.assert_array_equal(s.iterate(c.clone(), 2), batch.iterate([c.clone()], 2)[0])
        batch.close()
