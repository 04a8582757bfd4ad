"""Inputs at the edges of what the structured evaluation's own arithmetic
covers: the end of the range that its sine and cosine reduce themselves, one
variable, values below the normal float range, parameters that are finite in
FP64 only."""
import math

import numpy as np
import pytest

import paper_2410_22575_gb300 as cf
from paper_2410_22575_gb300 import workloads as W

from gpu_helpers import BOUND, Dev

pytestmark = pytest.mark.gpu


def _ackley_far(x, v):
    """H and H v of Ackley at points with a variable so large that
    exp(-0.2 sqrt(S/n)) is 0: (4 pi^2/n) exp(C/n) (diag(cos) - sin sin^T / n),
    the angles from the exact fractional parts."""
    n = x.shape[1]
    t = x - np.rint(x)
    s, c = np.sin(2 * math.pi * t), np.cos(2 * math.pi * t)
    k = 4 * math.pi ** 2 / n * np.exp(c.mean(1))
    H = k[:, None, None] * (np.eye(n)[None] * c[:, None, :] - s[:, :, None] * s[:, None, :] / n)
    return H, np.einsum("pij,pj->pi", H, v)


@pytest.mark.parametrize("n", [1, 2, 5, 64, 130])
def test_ackley_fp64_large_arguments(n):
    """|x| on both sides of 2^49 and 2^50, beyond which 4x + 1.5 * 2^52 is no
    longer rounded to an integer, and beyond which the units of x are whole
    turns; H v, Hessian and uneven request."""
    import torch

    far = [2.0 ** 47 + 0.25, 2.0 ** 48, 2.0 ** 49 - 0.25, 2.0 ** 49, 2.0 ** 49 + 0.5, 9e14 + 1, 2.0 ** 50 - 0.5,
           2.0 ** 50, 2.0 ** 51 + 1]
    far = np.array(far + [-t for t in far])
    b = W.make_batch(W.ACKLEY, n, len(far), seed=60 + n)
    b.x[np.arange(len(far)), np.arange(len(far)) % n] = far
    d = Dev(b, cf.FP64)
    H, Hv = _ackley_far(d.xh, d.vh)
    scale = np.sqrt((H * H).sum((1, 2)))
    out = d.hvp()
    assert np.all(np.linalg.norm(out - Hv, axis=1) <= BOUND[cf.FP64] * scale * np.linalg.norm(d.vh, axis=1))
    assert np.all(np.sqrt(((d.hessian() - H) ** 2).sum((1, 2))) <= BOUND[cf.FP64] * scale)
    plan = cf.RaggedPlan(cf.requests([W.ACKLEY] * len(far), [n] * len(far), np.arange(len(far)) * n), cf.FP64)
    packed = torch.empty_like(d.x)
    plan.run(d.x, d.v, packed)
    torch.cuda.synchronize()
    got = packed.cpu().numpy()
    assert np.all(np.linalg.norm(got - Hv, axis=1) <= BOUND[cf.FP64] * scale * np.linalg.norm(d.vh, axis=1))


def test_fletcher_powell_one_variable_hessian_many_points():
    """n = 1 in compensated FP32: the entry 2 J^2 + 2 r P, whose terms cancel at
    some points, is formed in FP64 and rounded once, at each of 200000 points;
    where a value is not finite it is what the dense method gives."""
    b = W.make_batch(W.FLETCHER_POWELL, 1, 200000, seed=9)
    b.x[5, 0], b.x[6, 0], b.x[7, 0] = np.nan, np.inf, -np.inf
    d = Dev(b, cf.FP32_COMP)
    H = d.hessian()[:, 0, 0]
    A, B, E = float(b.fp.A[0, 0]), float(b.fp.B[0, 0]), float(b.fp.E[0])
    x = d.xh[:, 0]
    with np.errstate(invalid="ignore"):
        s, c = np.sin(x), np.cos(x)
    ref = 2 * (A * c - B * s) ** 2 + 2 * (E - A * s - B * c) * (A * s + B * c)
    ok = np.isfinite(ref)
    assert np.all(np.isnan(H[~ok]))
    assert np.max(np.abs(H[ok] - ref[ok]) / np.abs(ref[ok])) <= BOUND[cf.FP32_COMP]
    for which in range(3):
        b = W.make_batch(W.FLETCHER_POWELL, 1, 300, seed=9)
        (b.fp.A, b.fp.B, b.fp.E)[which].flat[0] = np.inf
        d = Dev(b, cf.FP32_COMP)
        assert np.array_equal(d.hessian(), d.hessian(cfg=cf.Config(1, 1, 256)), equal_nan=True)


@pytest.mark.parametrize("n", [3, 13, 64, 70, 140])
@pytest.mark.parametrize("which", [0, 1])
def test_fletcher_powell_fp32_parameters_beyond_float(n, which):
    """An entry of A (B) finite in FP64 and infinite in FP32, in a column whose
    sin (cos) hides it from the residuals at one point: every entry is NaN
    there, as the dense method has it, whatever the column."""
    for j in (0, n // 2, n - 1):
        b = W.make_batch(W.FLETCHER_POWELL, n, 6, seed=80 + n)
        (b.fp.A, b.fp.B)[which][1, j] = 1e39
        b.x[2:4, j] = 0.0 if which == 0 else math.pi / 2
        d = Dev(b, cf.FP32_COMP)
        cfg = cf.Config(0, 0, 0, cf.SYMMETRIC, 0) if n >= 4 else cf.Config(2, 1, 256)
        for got, dense in ((d.hessian(), d.hessian(cfg=cfg)), (d.hvp(), d.hvp(cfg=cfg))):
            assert np.array_equal(np.isnan(got), np.isnan(dense)), j


@pytest.mark.parametrize("n", [5, 40, 140])
def test_fletcher_powell_fp32_subnormal_parameters(n):
    """A column of A and B whose floats are subnormal (rounded to 2^-149, a
    relative 2e-5 of 1e-40): its row of H v and its diagonal entry keep three
    digits."""
    j = n // 2
    b = W.make_batch(W.FLETCHER_POWELL, n, 20, seed=70 + n)
    b.fp.A[:, j] *= 1e-42  # |A|, |B| up to 100
    b.fp.B[:, j] *= 1e-42
    d = Dev(b, cf.FP32_COMP)
    Hv, _ = d.ref_hvp()
    H = d.ref_hessian()
    row, diag = d.hvp()[:, j], d.hessian()[:, j, j]
    assert np.max(np.abs(Hv[:, j])) > 0
    assert np.max(np.abs(row - Hv[:, j])) <= 1e-3 * np.max(np.abs(Hv[:, j]))
    assert np.max(np.abs(diag - H[:, j, j])) <= 1e-3 * np.max(np.abs(H[:, j, j]))
