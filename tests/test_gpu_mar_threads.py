"""FBP from several threads, each with a context of its own: rows of different
lengths, all of them above the 48 KB of shared memory that a block has without
asking for more.  Every call succeeds, with the image that it gives alone."""
import dataclasses
import threading

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


def _scan(pkg, K):
    geo = synth.Geometry(synth.FAN2D, 8, 8, 1, 4.0, 4.0, 0.75, 0.0, 0.0, 0.0, 570.0, 1040.0, 2, 2, 0.3, 0.0, 0.0, 1,
                         0.75 * 1040.0 / 570.0, K, synth.fan_pitch(24.0, 570.0, K), 0.25, 0.0)
    case = dataclasses.replace(synth.make_case("t3d"), geo=geo)
    d, _ = synth.measure(case, seed=1, noiseless=True)
    s = pkg.from_case(case)
    s.set_data(d.cuda())
    return s, s.log_sinogram()


def test_fbp_of_long_rows_in_two_threads(pkg):
    scans = [_scan(pkg, K) for K in (3072, 2048)]
    alone = [s.fbp(p) for s, p in scans]
    torch.cuda.synchronize()
    faults = []
    start = threading.Barrier(len(scans))

    def run(i):
        s, p = scans[i]
        start.wait()
        try:
            for n in range(3000):
                img = s.fbp(p)
                if n % 500 == 0 and not torch.equal(img, alone[i]):
                    faults.append(f"{p.shape[-1]} channels, call {n}: another image")
        except pkg.DeamError as e:
            faults.append(f"{p.shape[-1]} channels, call {n}: {e}")

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(scans))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not faults, faults
