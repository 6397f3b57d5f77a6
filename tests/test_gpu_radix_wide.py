"""Run starts of the radix sort where most keys of a window have no item: results against
the closed form for gaps of every kind (before the first key, between neighbours, after the
last, a whole window of zero digits), and the time the gaps may take."""
import numpy as np
import pytest
import torch

from oracle import g1
from tests.util import closed_form_limbs, msm_inputs

pytestmark = pytest.mark.gpu

pkg = pytest.importorskip("paper_2502_11660_gb300")


@pytest.mark.parametrize("edwards", [False, True])
@pytest.mark.parametrize("c", [5, 6, 9, 16, 20])
@pytest.mark.parametrize("n", [1, 255, 256, 257, 700])
def test_windows_of_few_keys(n, c, edwards):
    a, s, pts = msm_inputs(700, tag=72)
    a, s, pts = a[:n].copy(), s[:n], pts[:n]
    a[n // 2:] = 0                                   # zero digits: no key but 0
    a[n // 4:n // 2, 1:] = 0                         # only the low windows have keys
    a[n // 3:n // 2, 0] = (1 << (c - 1)) - (np.arange(n // 2 - n // 3) % 2).astype(np.uint32)   # the last two keys
    out = pkg.msm_g1(pkg.to_device(pts), pkg.to_device(a), c=c, scalar_bits=253, edwards=edwards, radix_sort=True)
    torch.cuda.synchronize()
    assert g1.from_limbs(pkg.to_host(out)) == closed_form_limbs(s, a)


def test_the_gaps_cost_no_more_than_the_counting_sort():
    """Zero scalars at c = 20: 13 windows of 2^19 keys without an item. The counting sort's
    head passes over its bins five times; the radix sort's, whose passes over 100 items are
    a dozen small launches, may take twice that, not a serial loop over the keys (4 times)."""
    n = 100
    _, _, pts = msm_inputs(700, tag=72)
    points = pkg.msm_points_prepare(pkg.to_device(pts[:n]))
    scalars = torch.zeros((n, 8), dtype=torch.int32, device="cuda")
    head = {}
    for radix in (False, True):
        kw = dict(c=20, scalar_bits=253, prepared=True, radix_sort=radix)
        ws = pkg.msm_g1_workspace(n, **kw)
        times = []
        for _ in range(8):
            pkg.msm_g1(points, scalars, workspace=ws, profile=True, **kw)
            times.append(pkg.profile_last()["head"])
        head[radix] = min(times[2:])
    assert head[True] < 2 * head[False], head
