"""The one-launch plan of a batch whose scans take one, two and four rays per turn of
the backprojection, side by side in every slab class: one iteration against each
scan's own.

Both add the same n samples to a voxel's sums, in another order: FP32 sums that differ
by 2 n 2^-24 of the sum of magnitudes at most.  With counts within a fifth of the
model's, delta / b~ and its logarithm then differ by less than 4 n 2^-24, and the image
by 1 / Z of that and a rounding."""
import dataclasses

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


def _case(nx, nz, V, R, dz, dx, K):
    geo = synth.Geometry(synth.HELICAL, nx, nx - 3, nz, dx, dx, dz, 0.0, 0.0, 0.0, 570.0, 1040.0, V, 96, 0.3,
                         0.2 * dz * 96, -0.1 * dz * V, R, 0.75 * 1040.0 / 570.0, K,
                         synth.fan_pitch(nx * dx / 2.0, 570.0, K), 0.25, 0.0)
    return dataclasses.replace(synth.make_case("t3d"), geo=geo)


@pytest.mark.parametrize("channels", [(7,), (17, 43), (50,), (2, 15, 40, 90)])
def test_rays_per_turn_in_a_batch(pkg, channels):
    gen = torch.Generator(device="cuda").manual_seed(7)
    scans, images = [], []
    for K in channels:
        for nz, dz, R in [(18, 0.75, 16), (13, 1.5, 11), (2, 0.75, 4), (1, 0.75, 1)]:
            g = pkg.from_case(_case(40, nz, 50, R, dz, 4.0, K))
            c = 0.3 + 0.2 * torch.rand(g.img_shape, generator=gen, device="cuda")
            _, counts = g.forward(c, want_l=False, want_g=True)
            g.set_data(counts * (0.8 + 0.4 * torch.rand(counts.shape, generator=gen, device="cuda")))
            scans.append(g)
            images.append(c)
    batch = pkg.DeamBatch(scans, autotune=False)
    got = [c.clone() for c in images]
    batch.iterate(got, 1)
    assert batch.info()["plan"] == "persistent"
    for g, c, x in zip(scans, images, got):
        geo = g.geo
        _, _, Z = g.backprojected_sums(c)
        want = c.clone()
        g.iterate(want, 1)
        # rays of a view, and rows, within a voxel of a column, at most (0.7: the nearest
        # columns' distance from the source over the axis')
        taps = 2.0 * geo.dx / (0.7 * geo.sid * geo.channel_pitch) + 1.0
        rows = min(geo.n_rows, 2.0 * geo.dz / (0.7 * 0.75) + 1.0)
        n = geo.n_views * taps * rows
        assert (want - c).abs().max() * Z > 0.01
        assert (x - want).abs().max() <= 4.0 * n * 2.0**-24 / Z + 2.0**-23 * want.abs().max()
    batch.close()
    for g in scans:
        g.close()
