"""Building an uneven plan takes time in proportion to its requests (no GPU)."""
import time

import numpy as np
import pytest

import paper_2410_22575_gb300 as cf


def _seconds(nreq, prec, fns):
    rng = np.random.Generator(np.random.PCG64(1))
    ns = rng.integers(2, 40, nreq)
    reqs = cf.requests(np.resize(fns, nreq), ns, np.concatenate([[0], np.cumsum(ns[:-1])]), [0] * nreq)
    best = 1e30
    for _ in range(3):
        t = time.perf_counter()
        h = cf.chessfad_ragged_plan_create(reqs, prec)
        best = min(best, time.perf_counter() - t)
        cf.chessfad_ragged_plan_destroy(h)
    return best


@pytest.mark.parametrize("prec", [cf.FP64, cf.FP32_COMP])
@pytest.mark.parametrize("fns", [[0, 1, 2], [2]])
def test_plan_time_is_not_quadratic(prec, fns):
    """Eight times the requests: 8 to 9 times the time, where walking a group's
    requests for every tile takes 64 times."""
    small, large = _seconds(25000, prec, fns), _seconds(200000, prec, fns)
    assert large <= 24 * small, (small, large)
