"""GPU parity of the four-warp window chains where their Weierstrass addition has a
special case: two windows' sums that differ by a point of order 2 (where the complete
formulas give (0 : 0 : 0)), equal, opposite or empty window sums, and windows of every
chain length. Exact affine points against the chord/tangent oracle."""
import numpy as np
import pytest
import torch

import synth
from oracle import fq, g1

pytestmark = pytest.mark.gpu

pkg = pytest.importorskip("paper_2502_11660_gb300")

T2 = (fq.P - 1, 0)   # the point (-1, 0) of order 2


def _run(points, scalars, c, **kw):
    pts = np.array([g1.to_limbs(p) for p in points], dtype=np.uint32)
    sc = np.stack([synth.int_to_limbs(k, 8) for k in scalars])
    out = pkg.msm_g1(pkg.to_device(pts), pkg.to_device(sc), c=c, **kw)
    torch.cuda.synchronize()
    return g1.from_limbs(pkg.to_host(out))


@pytest.mark.parametrize("c", [2, 5, 8])
@pytest.mark.parametrize("case", ["order_two_apart", "equal", "opposite", "order_two_only", "empty_low"])
def test_window_sums_with_special_cases(c, case):
    B = g1.random_point(11)                       # any curve point, outside the subgroup
    S1 = g1.mul(1 << c, B)                        # what the chain holds when S_0 is added
    C, k0 = {"order_two_apart": (g1.add(S1, T2), 1), "equal": (S1, 1), "opposite": (g1.neg(S1), 1),
             "order_two_only": (T2, 1), "empty_low": (S1, 0)}[case]
    want = g1.add(S1, g1.mul(k0, C))
    assert _run([B, C], [1 << c, k0], c) == want


@pytest.mark.parametrize("mode", [dict(), dict(edwards=True), dict(edwards=True, glv=True), dict(glv=True)])
@pytest.mark.parametrize("c", [2, 3, 7, 13])
def test_one_point_every_width(mode, c):
    for k in (0, 1, 2, (1 << c) - 1, 1 << (c + 1), fq.R - 1):
        assert _run([g1.G], [k], c, scalar_bits=253, **mode) == g1.mul(k, g1.G)
