"""padd_batch with many doublings: each warp puts its doublings off and does up to 32 of
them together, so batches where every, every other or almost no addition is one, at sizes
around a block and beyond one pass of the grid, against k G from the points' seeds."""
import numpy as np
import pytest
import torch

import synth
from oracle import fq

pytestmark = pytest.mark.gpu

pkg = pytest.importorskip("paper_2502_11660_gb300")


def _affine_points(seeds):
    """(n, 8) seeds -> [2][12][n] standard-form coordinates of seeds_i G."""
    p = pkg.g1_generator_mul(pkg.to_device(seeds))
    return p.t().reshape(2, 12, seeds.shape[0]).contiguous()


@pytest.mark.parametrize("n,every", [(1, 1), (31, 1), (129, 1), (129, 2), (19457, 3), (38912, 3), (38913, 3), (70001, 1), (150001, 2), (150001, 37)])
@pytest.mark.parametrize("form", ["standard", "montgomery"])
def test_doublings_among_additions(n, every, form):
    a, b = synth.scalars(41, n), synth.scalars(42, n)
    b[::every] = a[::every]
    acc_aff, q = _affine_points(a), _affine_points(b)
    acc = torch.zeros((4, 12, n), dtype=torch.int32, device="cuda")
    acc[:2] = acc_aff
    acc[2, 0] = acc[3, 0] = 1
    f = pkg.FORM_STANDARD
    if form == "montgomery":
        f = pkg.FORM_MONTGOMERY
        acc = torch.stack([pkg.fq_to_montgomery(x.contiguous()) for x in acc])
        q = torch.stack([pkg.fq_to_montgomery(x.contiguous()) for x in q])
    aff = pkg.xyzz_to_affine_batch(pkg.padd_batch(acc, q, form=f), form=f)
    if form == "montgomery":
        aff = torch.stack([pkg.fq_from_montgomery(x.contiguous()) for x in aff])
    sums = [(synth.limbs_to_int(x) + synth.limbs_to_int(y)) % fq.R for x, y in zip(a, b)]
    want = _affine_points(np.stack([synth.int_to_limbs(k, 8) for k in sums]))
    assert torch.equal(aff, want)
