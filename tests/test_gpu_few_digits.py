"""Scalars whose digits are mostly zero, at sizes whose pieces are long: results against the
closed form for both sorts, several window groups and batches (whose jobs' runs then need
more parts, and more merge levels, than uniform digits would), and the time they may take."""
import numpy as np
import pytest
import torch

import synth
from oracle import g1
from tests.util import closed_form_limbs

pytestmark = pytest.mark.gpu

pkg = pytest.importorskip("paper_2502_11660_gb300")

N = 1 << 17
_SETS: dict = {}


def point_set(edwards, glv, n=N):
    key = (edwards, glv, n)
    if key not in _SETS:
        seeds = synth.scalars(81, n)
        _SETS[key] = seeds, pkg.msm_points_prepare(pkg.g1_generator_mul(pkg.to_device(seeds)), edwards=edwards, glv=glv)
    return _SETS[key]


def scalars(kind, n):
    a = synth.scalars(82, n).copy()
    if kind == "ones":          # one run in one window
        a[:] = 0
        a[:, 0] = 1
    elif kind == "words":       # the low windows full, the others empty
        a[:, 1:] = 0
    elif kind == "half":        # about half the digits: either side of the rule
        a[: n // 2 + (n // 64 if n % 2 else 0)] = 0
    elif kind == "zero":
        a[:] = 0
    return a


@pytest.mark.parametrize("edwards,glv", [(False, False), (True, True)])
@pytest.mark.parametrize("radix", [False, True])
@pytest.mark.parametrize("kind", ["ones", "words", "half", "zero"])
@pytest.mark.parametrize("n,c", [(N, 5), (N, 9), (N - 1, 12)])
def test_few_nonzero_digits(n, c, kind, radix, edwards, glv):
    seeds, pts = point_set(edwards, glv)
    a = scalars(kind, n)
    out = pkg.msm_g1(pts[: n * (1 + glv)], pkg.to_device(a), c=c, scalar_bits=253, prepared=True, edwards=edwards,
                     glv=glv, radix_sort=radix)
    torch.cuda.synchronize()
    assert g1.from_limbs(pkg.to_host(out)) == closed_form_limbs(seeds[:n], a, key=("few", kind, n))


@pytest.mark.parametrize("groups", [2, 5])
@pytest.mark.parametrize("kind", ["ones", "words"])
def test_few_nonzero_digits_in_window_groups(kind, groups):
    """All nonzero digits are in the first group's windows."""
    seeds, pts = point_set(True, True)
    a = scalars(kind, N)
    pkg.msm_g1_set_schedule(17, groups=groups, edwards=True, glv=True)
    try:
        out = pkg.msm_g1(pts, pkg.to_device(a), c=9, scalar_bits=253, prepared=True, edwards=True, glv=True)
        torch.cuda.synchronize()
    finally:
        pkg.msm_g1_set_schedule(17, edwards=True, glv=True)
    assert g1.from_limbs(pkg.to_host(out)) == closed_form_limbs(seeds, a, key=("few", kind, N))


@pytest.mark.parametrize("edwards,glv", [(False, False), (True, True)])
def test_few_nonzero_digits_in_a_batch(edwards, glv):
    """A batch large enough for its longest pieces (48), and jobs around the numbers of items at
    which a run of ones takes its second part and its second tree level."""
    seeds, pts = point_set(edwards, glv, 1 << 19)
    sizes = [1 << 19, 1 << 19, 5, 6, 7, 24, 25, 47, 48, 49, 50, 383, 385, 1500, 3073, 20000]
    kinds = ["", ""] + ["ones"] * 14
    a = [scalars(k, n) for k, n in zip(kinds, sizes)]
    outs = pkg.msm_g1_batched([pts[: n * (1 + glv)] for n in sizes], [pkg.to_device(x) for x in a], scalar_bits=253,
                              prepared=True, edwards=edwards, glv=glv)
    torch.cuda.synchronize()
    for n, x, k, o in zip(sizes, a, kinds, outs):
        assert g1.from_limbs(pkg.to_host(o)) == closed_form_limbs(seeds[:n], x, key=("few", k, n)), n


def test_a_run_of_ones_uses_the_threads_it_can():
    """2^19 ones at c = 12: a tenth of the digits of uniform scalars, whose additions keep the
    multiply pipe busy; with enough pieces they take less than a quarter of that time (in
    pieces as long as the uniform digits' they take two fifths)."""
    n = 1 << 19
    seeds, pts = point_set(True, True, n)
    kw = dict(c=12, scalar_bits=253, prepared=True, edwards=True, glv=True)
    ws = pkg.msm_g1_workspace(n, **kw)
    took = {}
    for kind in ("", "ones"):
        sc = pkg.to_device(scalars(kind, n))
        times = []
        for _ in range(6):
            pkg.msm_g1(pts, sc, workspace=ws, profile=True, **kw)
            times.append(pkg.profile_last()["accumulate"])
        took[kind] = min(times[2:])
    assert took["ones"] < took[""] / 4, took
