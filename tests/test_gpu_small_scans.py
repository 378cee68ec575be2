"""Scans of few rays, thin volumes: what a call costs follows what it works on."""
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


def _scan(pkg, V, R, K, nx=160, nz=24, **kw):
    geo = synth.Geometry(synth.HELICAL, nx, nx, nz, 1.5, 1.5, 0.75, 0.0, 0.0, 0.0, 570.0, 1040.0, V, V, 0.3, 0.5 * R,
                         -0.25 * R, R, 0.75 * 1040.0 / 570.0, K, synth.fan_pitch(nx * 0.75, 570.0, K), 0.25, 0.0)
    return pkg.from_case(dataclasses.replace(synth.make_case("t3d"), geo=geo), **kw)


def _ms(f, n=9):
    f()
    times = []
    for _ in range(n):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    return sorted(times)[n // 2]


def test_penalty_follows_the_voxels(pkg):
    # R(c) reads the image alone: the same volume with 40 rays and with a million
    # takes the same time (half as long again is left for the clock's spread) and
    # has the same value up to the order of FP64 sums (1e-12)
    few, many = (_scan(pkg, *rays, penalty_lambda=3.0, penalty_delta=0.05) for rays in ((2, 1, 20), (360, 16, 200)))
    c = torch.rand(few.img_shape, generator=torch.Generator().manual_seed(4)).cuda()
    a, b = few.penalty(c), many.penalty(c)
    assert abs(a - b) <= 1e-12 * abs(b)
    assert _ms(lambda: few.penalty(c)) <= 1.5 * _ms(lambda: many.penalty(c))
    few.close()
    many.close()


def test_count_follows_the_rays(pkg):
    # the same rays through two slices and through 24: the count visits each ray once
    # (a quarter is left for the clock's spread)
    thin, thick = _scan(pkg, 360, 16, 500, nz=2), _scan(pkg, 360, 16, 500)
    assert 0 < thin.count_samples() < thick.count_samples()
    assert _ms(thin.count_samples, 25) <= 1.25 * _ms(thick.count_samples, 25)
    thin.close()
    thick.close()
