"""GPU parity of the bucket accumulation's pieces and their merges: one bucket per window
(equal scalars) cut into every number of parts at which the merge changes form (one
piece, the threads' sums, one tree block, two and three tree levels), beside buckets of
one point, for both sorts and both curve models, against the closed form."""
import numpy as np
import pytest
import torch

from oracle import g1
from tests.util import closed_form_limbs, msm_inputs

pytestmark = pytest.mark.gpu

pkg = pytest.importorskip("paper_2502_11660_gb300")


@pytest.mark.parametrize("edwards", [False, True])
@pytest.mark.parametrize("radix", [False, True])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 17, 19, 128, 130, 8192, 8194, 8400])
def test_one_bucket_of_many_parts(n, radix, edwards):
    a, s, pts = msm_inputs(8400, tag=71)
    a, s, pts = a[:n].copy(), s[:n], pts[:n]
    a[: max(1, n - 100 * (n > 1000))] = a[0]      # some buckets of one or two points beside it
    kw = dict(edwards=edwards, precomputed=False)
    k = n.bit_length() - 1
    pkg.msm_g1_set_schedule(k, 0, 2, 0, 0, 0, **kw)   # pieces of at most two points
    try:
        for c in (4, 12):                         # few and many buckets
            out = pkg.msm_g1(pkg.to_device(pts), pkg.to_device(a), c=c, scalar_bits=253, edwards=edwards,
                             radix_sort=radix)
            torch.cuda.synchronize()
            assert g1.from_limbs(pkg.to_host(out)) == closed_form_limbs(s, a)
    finally:
        pkg.msm_g1_set_schedule(k, **kw)


@pytest.mark.parametrize("edwards", [False, True])
def test_longest_pieces(edwards):
    """Runs around the longest piece the lists can hold (256)."""
    n = 1030
    a, s, pts = msm_inputs(8400, tag=71)
    a, s, pts = a[:n].copy(), s[:n], pts[:n]
    for lo, hi in ((0, 255), (255, 511), (511, 768), (768, 1025)):   # 255, 256, 257, 257 equal scalars
        a[lo:hi] = a[lo]
    k = n.bit_length() - 1
    pkg.msm_g1_set_schedule(k, 0, 256, 0, 0, 0, edwards=edwards)
    try:
        out = pkg.msm_g1(pkg.to_device(pts), pkg.to_device(a), c=9, scalar_bits=253, edwards=edwards)
        torch.cuda.synchronize()
        assert g1.from_limbs(pkg.to_host(out)) == closed_form_limbs(s, a)
    finally:
        pkg.msm_g1_set_schedule(k, edwards=edwards)


@pytest.mark.parametrize("edwards", [False, True])
@pytest.mark.parametrize("c,reduce_log2", [(2, 8), (5, 8), (8, 8), (8, 13), (11, 8), (11, 12), (11, 20), (14, 10), (14, 17)])
def test_bucket_reduction_geometries(edwards, c, reduce_log2):
    """Segments of one to hundreds of buckets, most of them empty, in every split over blocks."""
    n = 300
    a, s, pts = msm_inputs(8400, tag=71)
    a, s, pts = a[:n], s[:n], pts[:n]
    k = n.bit_length() - 1
    pkg.msm_g1_set_schedule(k, 0, 0, 0, reduce_log2, 0, edwards=edwards)
    try:
        out = pkg.msm_g1(pkg.to_device(pts), pkg.to_device(a), c=c, scalar_bits=253, edwards=edwards)
        torch.cuda.synchronize()
        assert g1.from_limbs(pkg.to_host(out)) == closed_form_limbs(s, a)
    finally:
        pkg.msm_g1_set_schedule(k, edwards=edwards)
