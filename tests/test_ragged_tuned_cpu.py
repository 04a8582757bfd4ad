"""An uneven plan of the dense evaluation as tuned, on the host: the arguments'
checks, and the default configuration where nothing was tuned (no GPU)."""
import ctypes

import numpy as np
import pytest

import paper_2410_22575_gb300 as cf


def test_validation():
    lib, h = cf.load(), ctypes.c_void_p()
    r = cf.requests([0], [4], [0])
    assert lib.chessfad_ragged_plan_create_tuned(r.ctypes.data, 1, 5, ctypes.byref(h)) == -7
    assert lib.chessfad_ragged_plan_create_tuned(None, 3, 1, ctypes.byref(h)) == -5
    assert lib.chessfad_ragged_plan_create_tuned(r.ctypes.data, 1, 1, None) == -5
    bad = cf.requests([0], [513], [0])
    assert lib.chessfad_ragged_plan_create_tuned(bad.ctypes.data, 1, 1, ctypes.byref(h)) == -2
    with pytest.raises(ValueError, match="csize"):
        cf.RaggedPlan(r, cf.FP64, csize=8, tuned=True)


@pytest.mark.parametrize("prec,csize", [(cf.FP64, 8), (cf.FP32_COMP, 16)])
def test_untuned_groups_take_the_defaults(prec, csize):
    """Sizes of a range that nothing in the process tunes without a GPU: the
    plan is the one of the default chunk size."""
    import torch

    if torch.cuda.is_available():
        pytest.skip("the table may hold tuned entries")
    rng = np.random.Generator(np.random.PCG64(2))
    fns, ns = rng.integers(0, 3, 500), rng.integers(1, 300, 500)
    r = cf.requests(fns, ns, np.concatenate([[0], np.cumsum(ns[:-1])]), [0] * 500)
    h, ref = cf.chessfad_ragged_plan_create_tuned(r, prec), cf.chessfad_ragged_plan_create(r, prec, csize)
    assert cf.chessfad_ragged_plan_info(h) == cf.chessfad_ragged_plan_info(ref)
    for p in (h, ref):
        cf.chessfad_ragged_plan_destroy(p)
