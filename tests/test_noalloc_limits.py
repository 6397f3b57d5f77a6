"""Which requests msm_g1_noalloc takes: with c = 0 every one of up to 2^16 points, at a narrower
window where the default one does not fit its scratch, and none beyond what any width fits."""
import ctypes

import pytest

import paper_2502_11660_gb300 as pkg

MODELS = [0, pkg.EDWARDS, pkg.GLV, pkg.EDWARDS | pkg.GLV]
SCRATCH = 64 << 20


def too_large(n, flags, signed, c=0):
    """Whether the size check refuses the request (it comes before any look at the points)."""
    o = pkg.MsmOpts(c, signed, 0, flags, 0)
    rc = pkg.lib().msm_g1_noalloc(None, None, n, ctypes.c_void_p(16), ctypes.byref(o))
    assert rc != 0
    return rc == -1 and "bytes of scratch" in pkg.last_error()


@pytest.mark.parametrize("model", MODELS)
@pytest.mark.parametrize("prepared", [0, 1])
@pytest.mark.parametrize("signed", [0, 1])
def test_sizes_that_fit(model, prepared, signed):
    for n in (1, 4095, 4096, 1 << 15, 50000, 65535, 1 << 16):
        assert not too_large(n, model | prepared, signed), n


@pytest.mark.parametrize("model,n", [(0, 102500), (pkg.EDWARDS, 86200), (pkg.GLV, 90900),
                                     (pkg.EDWARDS | pkg.GLV, 75500)])
def test_sizes_just_beyond(model, n):
    def narrowest(n):
        return min(pkg.lib().msm_g1_workspace_bytes(n, ctypes.byref(pkg.MsmOpts(c, 1, 0, model, 0))) for c in range(4, 18))

    assert narrowest(n) > SCRATCH >= narrowest(n - 1000)   # no width fits n, one fits a little less
    assert too_large(n, model, 1) and not too_large(n - 1000, model, 1)


def test_an_explicit_width_is_not_narrowed():
    n = 60000
    need = pkg.lib().msm_g1_workspace_bytes(n, ctypes.byref(pkg.MsmOpts(13, 1, 0, 0, 0)))
    assert need > SCRATCH and too_large(n, 0, 1, c=13)
    assert not too_large(n, 0, 1)


@pytest.mark.gpu
@pytest.mark.parametrize("radix", [False, True])
@pytest.mark.parametrize("edwards,glv,n", [(False, False, 80000), (True, True, 66000)])
def test_narrowed_calls(edwards, glv, n, radix):
    import torch

    import synth
    from oracle import g1
    from tests.util import closed_form_limbs
    flags = pkg._model_flags(edwards, glv) | (pkg.RADIX_SORT if radix else 0)
    default = pkg.MsmOpts(pkg.msm_g1_default_c(n, True, edwards, glv), 1, 253, flags, 0)
    assert pkg.lib().msm_g1_workspace_bytes(n, ctypes.byref(default)) > SCRATCH   # the narrower width it is
    seeds, a = synth.scalars(95, n), synth.scalars(96, n)
    points, scalars = pkg.g1_generator_mul(pkg.to_device(seeds)), pkg.to_device(a)
    out = torch.full((24,), -1, dtype=torch.int32, device="cuda")
    o = pkg.MsmOpts(0, 1, 253, flags, torch.cuda.current_stream().cuda_stream)
    for _ in range(2):
        rc = pkg.lib().msm_g1_noalloc(ctypes.c_void_p(points.data_ptr()), ctypes.c_void_p(scalars.data_ptr()), n,
                                      ctypes.c_void_p(out.data_ptr()), ctypes.byref(o))
        assert rc == 0, pkg.last_error()
        torch.cuda.synchronize()
        assert g1.from_limbs(pkg.to_host(out)) == closed_form_limbs(seeds, a, key=("narrow", n))
