"""The plan of a batch does not depend on widths and piece lengths installed for single calls
(its workspace, which every part of the plan enters, stays the same)."""
import ctypes

import pytest

import paper_2502_11660_gb300 as pkg
from paper_2502_11660_gb300 import autotune


def batch_bytes(sizes, c=0, **kw):
    jobs = (pkg.MsmJob * len(sizes))()
    for job, n in zip(jobs, sizes):
        job.n, job.c = n, c
    return pkg.lib().msm_g1_batched_workspace_bytes(jobs, len(sizes), ctypes.byref(pkg._opts(0, prepared=True, **kw)))


@pytest.mark.parametrize("edwards,glv", [(False, False), (True, True)])
def test_installed_entries_are_for_single_calls(edwards, glv):
    mode = dict(edwards=edwards, glv=glv)
    sizes = [1 << 10, 3000, 1 << 14, 70000]
    built_in = batch_bytes(sizes, **mode)
    single = [pkg.msm_g1_schedule(n, **mode) for n in sizes]
    try:
        autotune.install([13] * 20, **mode)
        for k in range(10, 17):
            pkg.msm_g1_set_schedule(k, c=13, chunk=8, reduce_log2=17, **mode)
        assert [pkg.msm_g1_schedule(n, **mode)["c"] for n in sizes] == [13] * 4
        assert batch_bytes(sizes, **mode) == built_in
        assert batch_bytes(sizes, c=13, **mode) != built_in   # a job's own width still counts
    finally:
        autotune.clear(**mode)
        autotune.clear_schedule(**mode)
    assert [pkg.msm_g1_schedule(n, **mode) for n in sizes] == single
