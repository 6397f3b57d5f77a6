"""Edges of the merges and of the bucket reduction: one bucket of exactly as many parts as one
more would send down another path, and bit sums in several slices per bit."""
import numpy as np
import pytest
import torch

import synth
from oracle import g1
from tests.util import closed_form_limbs

pytestmark = pytest.mark.gpu

pkg = pytest.importorskip("paper_2502_11660_gb300")

N = 20000
_SETS: dict = {}


def point_set(edwards):
    if edwards not in _SETS:
        seeds = synth.scalars(97, N)
        _SETS[edwards] = seeds, pkg.msm_points_prepare(pkg.g1_generator_mul(pkg.to_device(seeds)), edwards=edwards)
    return _SETS[edwards]


@pytest.mark.parametrize("edwards", [False, True])
@pytest.mark.parametrize("others", [0, 100])
@pytest.mark.parametrize("parts", [2, 3, 8, 9, 64, 65, 4096, 4097])
def test_parts_of_one_bucket(parts, others, edwards):
    """Pieces of two: 2 * parts equal scalars, beside `others` of their own. A thread takes up to
    2 parts at c = 4 and 8 at c = 12, a block 64; beyond 64 there are two levels of blocks, beyond
    4096 three."""
    seeds, pts = point_set(edwards)
    n = 2 * parts + others
    a = synth.scalars(98, n).copy()
    a[others:] = a[others]
    k = n.bit_length() - 1
    pkg.msm_g1_set_schedule(k, chunk=2, edwards=edwards)
    try:
        for c in (4, 12):
            out = pkg.msm_g1(pts[:n], pkg.to_device(a), c=c, scalar_bits=253, prepared=True, edwards=edwards)
            torch.cuda.synchronize()
            assert g1.from_limbs(pkg.to_host(out)) == closed_form_limbs(seeds[:n], a, key=("parts", n))
    finally:
        pkg.msm_g1_set_schedule(k, edwards=edwards)


@pytest.mark.parametrize("edwards", [False, True])
@pytest.mark.parametrize("n", [40, 1500, N])             # mostly empty buckets to full ones
@pytest.mark.parametrize("bits", [8, 14, 24, 40, 90])
@pytest.mark.parametrize("c", [9, 12, 14, 16])
def test_bit_sums_in_slices(c, bits, n, edwards):
    """One to eleven windows: each bit's sum is cut into 16 to 2 slices, over segments of 1 to 8
    buckets, summed by one lane or two, and the slices of up to 256 points by 128 threads first."""
    seeds, pts = point_set(edwards)
    a = synth.scalars(99, n).copy()
    for w in range(8):
        keep = min(32, max(0, bits - 32 * w))
        a[:, w] &= np.uint32((1 << keep) - 1)
    out = pkg.msm_g1(pts[:n], pkg.to_device(a), c=c, scalar_bits=bits, prepared=True, edwards=edwards)
    torch.cuda.synchronize()
    assert g1.from_limbs(pkg.to_host(out)) == closed_form_limbs(seeds[:n], a, key=("slices", n, bits))
