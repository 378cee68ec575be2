"""What names the kernels that a scan runs: the plan query checks its arguments, and
the benchmark's names follow the plan (single slices have a kernel of their own, and
figures captured on one plan are not another's)."""
import ctypes as C

import pytest


@pytest.fixture(scope="module")
def pkg():
    from paper_2202_00116_gb300 import build
    build.build()
    import paper_2202_00116_gb300 as p
    return p


def test_plan_query_rejects_null(pkg):
    plan = pkg.deam_plan()
    assert pkg.lib().deam_kernel_plan(None, C.byref(plan)) == pkg.DEAM_ERR_ARG
    assert b"null" in pkg.lib().deam_last_error().lower()


def test_names_follow_the_plan():
    import bench
    plans = [dict(fwd_rows=r, bwd_slab=s, bwd_groups=g, bwd_rays=n)
             for r, s, g, n in [(1, 1, 8, 1), (1, 1, 16, 1), (8, 16, 1, 4), (4, 16, 2, 4), (4, 16, 4, 4), (4, 11, 4, 4)]]
    names = [bench.kernel_name("backproject", p) for p in plans]
    assert len(set(names)) == len(names)
    assert names[0].startswith("bwd_slice_kernel")
    assert bench.kernel_name("forward", plans[0]) != bench.kernel_name("forward", plans[2])
    # the captures are of the full-size scan's plan
    assert {bench.kernel_name(s, plans[2]) for s in ("forward", "backproject")} == set(bench.DRAM_BYTES_PER_SAMPLE)
    assert set(bench.L1_BUSY) == set(bench.DRAM_BYTES_PER_SAMPLE)
