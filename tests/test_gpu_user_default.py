"""The default H v of a user function where it could differ from the methods by
rows."""
import numpy as np
import pytest

import paper_2410_22575_gb300 as cf
from paper_2410_22575_gb300 import workloads as W

from test_gpu_user import PLAIN, SYM, Case, user_fn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [cf.FP64, cf.FP32_COMP])
def test_first_and_zeroth_powers_are_exact(prec):
    """pow(u, 0) is 1, the derivative of pow(u, 1) is 1 and, in FP32, pow(u, 1) is
    u (CUDA's double pow(x, 1.0) is not x at 4 % of x): every entry of this
    Hessian is 0 or 1 and, with whole v, every product a whole number."""
    import torch

    src = """template <class R, class X> R powers(const X &x, int n, const double *p)
    {
        R f = 0.0;
        for (int k = 0; k < n; ++k) {
            R a = pow(x[k], 1.0);
            if ((p[0] != 0.0 && a != x[k]) || pow(x[k], 0.0) != 1.0) f += 1e3 * x[k] * x[k];
            f += pow(x[k], 0.0) * x[k];
            if (k + 1 < n) f += a * x[k + 1];
        }
        return f;
    }"""
    f = cf.UserFunction(src, "powers", 8, prec)
    rng = np.random.Generator(np.random.PCG64(5))
    n = 30
    dt = torch.float64 if prec == cf.FP64 else torch.float32
    x = torch.tensor(rng.uniform(0.1, 5, (300, n)), dtype=dt, device="cuda")
    v = torch.tensor(rng.integers(-50, 51, (300, n)), dtype=dt, device="cuda")
    p = torch.tensor([float(prec == cf.FP32_COMP)], dtype=torch.float64, device="cuda")
    H = np.eye(n, k=1) + np.eye(n, k=-1)
    ref = v.double().cpu().numpy() @ H
    for cfg in (None, PLAIN, SYM):
        assert np.array_equal(f.hvp(x, v, p, cfg=cfg).double().cpu().numpy(), ref), cfg
    assert np.array_equal(f.hessian(x, p).double().cpu().numpy(), np.broadcast_to(H, (300, n, n)))


@pytest.mark.parametrize("prec", [cf.FP64, cf.FP32_COMP])
def test_powers_that_are_not_finite(prec):
    """Zero, negative, huge and tiny arguments of pow at whole and other
    exponents: the default product has the NaN and Inf of the plain method."""
    import torch

    src = """template <class R, class X> R mixed_powers(const X &x, int n, const double *p)
    { R f = 0.0; for (int k = 0; k < n; ++k) f += pow(x[k], p[k]) * (1.0 + x[0]); return f; }"""
    f = cf.UserFunction(src, "mixed_powers", 4, prec)
    dt = torch.float64 if prec == cf.FP64 else torch.float32
    big = 1e200 if prec == cf.FP64 else 1e30
    powers = [0.0, 1.0, 1.5, 2.0, 3.0, -1.0, 0.5, 40.0]
    n = len(powers)
    rng = np.random.Generator(np.random.PCG64(6))
    x = rng.uniform(0.1, 5, (48, n))
    for k, val in enumerate((0.0, -0.0, -2.0, big, 1 / big, np.inf)):
        x[8 * k + np.arange(8), np.arange(8)] = val
    x = torch.tensor(x, dtype=dt, device="cuda")
    v = torch.tensor(rng.uniform(-1, 1, (48, n)), dtype=dt, device="cuda")
    p = torch.tensor(powers, dtype=torch.float64, device="cuda")
    got, ref = (f.hvp(x, v, p, cfg=c).double().cpu().numpy() for c in (None, PLAIN))
    assert np.array_equal(np.isfinite(got), np.isfinite(ref))
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    ok = np.isfinite(ref)
    scale = np.max(np.abs(np.where(ok, ref, 0)), axis=1, keepdims=True) * np.ones_like(ref)
    assert np.all(np.abs(got - ref)[ok] <= (4e-12 if prec == cf.FP64 else 4e-5) * scale[ok])


def test_fp32_sums_over_the_direction_are_compensated():
    """f = (sum x)^2 / 2, every entry of H is 1: each row of H v is sum v as a
    compensated sum gives it, |error| <= 2u |sum v| + n^2 u^2 sum |v|."""
    import torch

    src = """template <class R, class X> R square_sum(const X &x, int n, const double *p)
    { R s = 0.0; for (int k = 0; k < n; ++k) s += x[k]; return 0.5 * s * s; }"""
    f = cf.UserFunction(src, "square_sum", 8, cf.FP32_COMP)
    u = 2.0 ** -24
    rng = np.random.Generator(np.random.PCG64(3))
    for n in (3, 64, 130, 512):
        x = torch.tensor(rng.uniform(-1, 1, (200, n)), dtype=torch.float32, device="cuda")
        v = torch.tensor(rng.uniform(-1, 1, (200, n)), dtype=torch.float32, device="cuda")
        vd = v.double().cpu().numpy()
        ref = vd.sum(1)
        err = np.abs(f.hvp(x, v).double().cpu().numpy() - ref[:, None]).max(1)
        assert np.all(err <= 2 * u * np.abs(ref) + n * n * u * u * np.abs(vd).sum(1)), n


@pytest.mark.parametrize("fn", [W.ROSENBROCK, W.ACKLEY, W.FLETCHER_POWELL, W.MIX])
@pytest.mark.parametrize("n,batch", [(5, 400), (19, 200), (64, 64), (200, 12)])
def test_fp32_default_is_as_accurate_as_the_symmetric_method(fn, n, batch):
    """Root mean square error over the batch, normalised by |H|_F |v|_2; 1.1
    allows for the different order of the sums."""
    f, k = user_fn(fn, 8, cf.FP32_COMP), Case(fn, n, batch, 300 + n, cf.FP32_COMP)
    rms = [np.sqrt(np.mean(k.hvp_err(f.hvp(k.x, k.v, k.params, cfg=c)) ** 2)) for c in (None, SYM)]
    assert rms[0] <= 1.1 * rms[1], rms


@pytest.mark.parametrize("prec", [cf.FP64, cf.FP32_COMP])
def test_source_that_names_the_number_type(prec):
    """A helper on chessfad::user::Num<T, C>, which takes the rows' numbers only:
    the handle is created and its default product is the symmetric method's."""
    src = """template <class T, int C> __device__ chessfad::user::Num<T, C> cube(const chessfad::user::Num<T, C> &u)
    { return u * u * u; }
    template <class R, class X> R cubes(const X &x, int n, const double *p)
    { R f = 0.0; for (int k = 0; k < n; ++k) f += cube(x[k]) * x[0]; return f; }"""
    f, k = cf.UserFunction(src, "cubes", 4, prec), Case(W.ROSENBROCK, 11, 50, 3, prec)
    out = f.hvp(k.x, k.v).double().cpu().numpy()
    assert np.array_equal(out, f.hvp(k.x, k.v, cfg=cf.Config(0, 0, 0, cf.SYMMETRIC, 32)).double().cpu().numpy())
    x, v = k.xh, k.vh
    H = np.zeros((50, 11, 11))
    i = np.arange(11)
    H[:, i, i] += 6 * x * x[:, :1]
    H[:, 0, :] += 3 * x ** 2
    H[:, :, 0] += 3 * x ** 2
    ref = np.einsum("pij,pj->pi", H, v)
    scale = np.sqrt((H * H).sum((1, 2))) * np.linalg.norm(v, axis=1)
    assert np.max(np.linalg.norm(out - ref, axis=1) / scale) <= (1e-12 if prec == cf.FP64 else 1e-5)
