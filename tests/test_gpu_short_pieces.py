"""An installed piece length far below the buckets' runs: every bucket is cut into many
parts. Results against the closed form where the parts of a bucket are put together by a
thread, by blocks and by both, and the time that putting them together may take."""
import pytest
import torch

import synth
from oracle import g1
from tests.util import closed_form_limbs

pytestmark = pytest.mark.gpu

pkg = pytest.importorskip("paper_2502_11660_gb300")

N = 1 << 16
_SETS: dict = {}


def point_set(edwards):
    if edwards not in _SETS:
        seeds = synth.scalars(91, N)
        _SETS[edwards] = seeds, pkg.msm_points_prepare(pkg.g1_generator_mul(pkg.to_device(seeds)), edwards=edwards)
    return _SETS[edwards]


@pytest.mark.parametrize("edwards", [False, True])
@pytest.mark.parametrize("heavy", [0, 400, 20000])     # equal scalars beside the uniform ones
@pytest.mark.parametrize("chunk,c", [(2, 7), (2, 9), (2, 12), (3, 10), (7, 12), (30, 9)])
def test_buckets_of_many_parts(chunk, c, heavy, edwards):
    seeds, pts = point_set(edwards)
    a = synth.scalars(92, N).copy()
    a[:heavy] = a[0]
    pkg.msm_g1_set_schedule(16, chunk=chunk, edwards=edwards)
    try:
        out = pkg.msm_g1(pts, pkg.to_device(a), c=c, scalar_bits=253, prepared=True, edwards=edwards)
        torch.cuda.synchronize()
    finally:
        pkg.msm_g1_set_schedule(16, edwards=edwards)
    assert g1.from_limbs(pkg.to_host(out)) == closed_form_limbs(seeds, a, key=("short", heavy))


def test_pieces_of_two_points():
    """c = 12: 45056 buckets of 16 parts each. Putting them together takes 15 additions of 14
    field products where the built-in pieces take 32 of 10 per bucket: at most about twice the
    products in all, so three times the time (a block for each bucket took eight times)."""
    seeds, pts = point_set(False)
    a = pkg.to_device(synth.scalars(92, N))
    took = {}
    for chunk in (0, 2):
        pkg.msm_g1_set_schedule(16, chunk=chunk)
        try:
            kw = dict(c=12, scalar_bits=253, prepared=True)
            ws = pkg.msm_g1_workspace(N, **kw)
            times = []
            for _ in range(6):
                pkg.msm_g1(pts, a, workspace=ws, profile=True, **kw)
                times.append(sum(pkg.profile_last().values()))
            took[chunk] = min(times[2:])
        finally:
            pkg.msm_g1_set_schedule(16)
    assert took[2] < 3 * took[0], took
