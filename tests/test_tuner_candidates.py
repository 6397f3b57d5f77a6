"""The widths the autotuner times include those the library takes by itself, with and without
other widths installed, so a tuned table never holds less than the best of both."""
import pytest

import paper_2502_11660_gb300 as pkg
from paper_2502_11660_gb300 import autotune

MODES = [(False, False), (True, False), (False, True), (True, True)]


@pytest.mark.parametrize("edwards,glv", MODES)
def test_built_in_widths_are_timed(edwards, glv):
    built_in = {k: pkg.msm_g1_default_c(1 << k, True, edwards, glv) for k in range(23)}
    try:
        for installed in (0, 9, 13):
            autotune.install([installed] * 32, edwards=edwards, glv=glv)
            for k, c in built_in.items():
                cs = autotune.candidates(k, glv, edwards=edwards)
                assert c in cs, (k, c, cs)
                assert pkg.msm_g1_default_c(1 << k, True, edwards, glv) in cs   # the one in use
                assert len(cs) <= 9 and all(2 <= x <= 20 for x in cs)
    finally:
        autotune.clear(edwards=edwards, glv=glv)


def test_fixed_base_widths():
    assert autotune.candidates(16, precomputed=True) == list(autotune.PRECOMPUTED_C)
    assert autotune.candidates(12, precomputed=True) == [6, 7, 8, 9, 10]
