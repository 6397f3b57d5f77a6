"""The workspace a call of n points asks for holds the calls of fewer points too, up to the
sixth by which a layout falls where the pieces of its bucket runs become longer."""
import ctypes

import pytest

import paper_2502_11660_gb300 as pkg

SIZES = sorted({int(2 ** (k / 24)) for k in range(24 * 24)} |
               {s for k in range(1, 25) for s in ((1 << k) - 1, 1 << k, (1 << k) + 1)})


def need(n, **kw):
    return pkg.lib().msm_g1_workspace_bytes(n, ctypes.byref(pkg._opts(0, **kw)))


def worst_fall(**kw):
    largest, worst = 0, 1.0
    for n in SIZES:
        b = need(n, **kw)
        largest = max(largest, b)
        worst = max(worst, largest / b)
    return worst


@pytest.mark.parametrize("edwards", [False, True])
@pytest.mark.parametrize("glv", [False, True])
@pytest.mark.parametrize("kw", [dict(), dict(prepared=True), dict(radix_sort=True), dict(scalar_bits=253),
                                dict(scalar_bits=64)])
def test_need_over_sizes(kw, edwards, glv):
    assert worst_fall(edwards=edwards, glv=glv, **kw) < 1.25


def test_need_with_an_installed_table():
    from paper_2502_11660_gb300 import autotune
    try:
        autotune.install([0] * 10 + [16, 9, 14, 6, 10, 10])
        assert worst_fall(scalar_bits=253) < 1.25
    finally:
        autotune.clear()
