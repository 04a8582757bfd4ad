"""The structured evaluation (calls that name neither a chunk size nor a
method) against the oracle and against the dense symmetric method: sizes at
the edges of its lane groups, shared-memory tiles and pair limits, batches
that leave a ragged last CTA, and non-finite or overflowing points, which must
give what the dense method gives."""
import numpy as np
import pytest

import paper_2410_22575_gb300 as cf
from paper_2410_22575_gb300 import workloads as W

from gpu_helpers import BOUND, Dev, hessian_err, hvp_err

pytestmark = pytest.mark.gpu

FNS = [W.ROSENBROCK, W.ACKLEY, W.FLETCHER_POWELL]
PRECS = [cf.FP64, cf.FP32_COMP]


@pytest.mark.parametrize("fn", FNS)
@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("n,batch", [(1, 700), (2, 1), (2, 3001), (3, 257), (4, 130), (7, 1000), (8, 33), (9, 70),
                                     (16, 5), (31, 77), (33, 40), (64, 333), (65, 9), (127, 5), (129, 3), (200, 3),
                                     (257, 2), (511, 2), (512, 1)])
def test_hvp_sizes(fn, prec, n, batch):
    d = Dev(W.make_batch(fn, n, batch, seed=2000 + n), prec)
    out = d.hvp()
    e = hvp_err(d, out)
    assert e.max() <= BOUND[prec], (e.max(), np.median(e))
    assert np.array_equal(out, d.hvp())


@pytest.mark.parametrize("fn", FNS)
@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("n,batch", [(1, 700), (2, 1), (2, 3001), (3, 257), (4, 130), (7, 600), (16, 5), (17, 77),
                                     (33, 40), (63, 7), (64, 30), (65, 9), (127, 5), (128, 2), (129, 3), (200, 3),
                                     (511, 1), (512, 1)])
def test_hessian_sizes(fn, prec, n, batch):
    d = Dev(W.make_batch(fn, n, batch, seed=3000 + n), prec)
    H = d.hessian()
    e = hessian_err(d, H)
    assert e.max() <= BOUND[prec], (e.max(), np.median(e))
    assert np.array_equal(H, np.swapaxes(H, 1, 2))
    assert np.array_equal(H, d.hessian())


def _same(a, b, bound, scale):
    """Equal NaN and Inf entries, finite entries within bound * scale."""
    assert np.array_equal(np.isnan(a), np.isnan(b))
    inf = np.isinf(b)
    assert np.array_equal(np.isinf(a), inf) and np.array_equal(a[inf], b[inf])
    ok = np.isfinite(b)
    assert np.all(np.abs(a[ok] - b[ok]) <= bound * scale)


@pytest.mark.parametrize("fn", FNS)
@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("n", [2, 3, 5, 21, 64, 300])
def test_non_finite_points_equal_the_dense_method(fn, prec, n):
    """NaN and Inf in x, in v and in both, v = 0 beside them, x at the origin
    (Ackley's square root) and x whose squares overflow: the default call
    against the dense method it stands for (plain below n = 4)."""
    bad = [np.nan, np.inf, -np.inf]
    huge = 1e30 if prec == cf.FP32_COMP else 1e200
    b = W.make_batch(fn, n, 24, seed=77 + n)
    for k, val in enumerate(bad):
        b.x[k, n // 2] = val
        b.x[3 + k, n - 1] = val
        b.v[6 + k, n // 2] = val
        b.x[9 + k, 0] = val
        b.v[9 + k, n - 1] = bad[(k + 1) % 3]
        b.x[18 + k, 0] = val
        b.v[18 + k] = 0.0
    b.v[12, 0], b.v[12, n - 1] = np.inf, -np.inf
    b.x[13] = 0.0
    if fn != W.FLETCHER_POWELL:  # sin and cos of huge arguments: compared through Rosenbrock and Ackley
        b.x[14, n // 2] = huge
        b.x[15, 0] = b.x[15, n - 1] = -huge
        b.x[16, n - 1] = huge
        b.x[17, n - 2] = huge
    d = Dev(b, prec)
    dense = d.hvp(cfg=cf.Config(0, 0, 0, cf.SYMMETRIC, 0) if n >= 4 else cf.Config(2, 1, 256))
    got = d.hvp()
    fine = np.isfinite(dense)
    scale = np.max(np.abs(np.where(fine, dense, 0.0)), axis=1, keepdims=True) * np.ones_like(dense)
    tol = 4e-12 if prec == cf.FP64 else 4e-5
    _same(got, dense, tol, scale[fine])
    dense = d.hessian(cfg=cf.Config(0, 0, 0, cf.SYMMETRIC, 0) if n >= 4 else cf.Config(2, 1, 256))
    got = d.hessian()
    fine = np.isfinite(dense)
    scale = np.max(np.abs(np.where(fine, dense, 0.0)), axis=(1, 2), keepdims=True) * np.ones_like(dense)
    _same(got, dense, tol, scale[fine])


@pytest.mark.parametrize("prec", PRECS)
def test_non_finite_parameters_equal_the_dense_method(prec):
    import torch

    for which in range(3):
        b = W.make_batch(W.FLETCHER_POWELL, 13, 50, seed=5)
        (b.fp.A, b.fp.B, b.fp.E)[which].flat[7] = np.inf
        d = Dev(b, prec)
        dense = d.hvp(cfg=cf.Config(0, 0, 0, cf.SYMMETRIC, 0))
        assert np.array_equal(np.isnan(d.hvp()), np.isnan(dense)) and np.all(~np.isfinite(dense))
        Hd, H = d.hessian(cfg=cf.Config(0, 0, 0, cf.SYMMETRIC, 0)), d.hessian()
        assert np.array_equal(np.isnan(H), np.isnan(Hd))
        assert np.array_equal(np.isinf(H), np.isinf(Hd)) and np.all(~np.isfinite(Hd))


@pytest.mark.parametrize("fn", FNS)
def test_points_are_independent(fn):
    """A permuted batch gives the permuted outputs bit for bit, also beside a
    non-finite point; an offset, 8-byte aligned view gives the same values."""
    import torch

    b = W.make_batch(fn, 19, 300, seed=8)
    b.x[100, 3] = np.nan
    d = Dev(b, cf.FP64)
    a = d.hvp()
    perm = np.random.Generator(np.random.PCG64(1)).permutation(300)
    dp = Dev(W.Batch("p", fn, 19, b.x[perm], b.v[perm], b.fp), cf.FP64)
    assert np.array_equal(dp.hvp(), a[perm], equal_nan=True)
    flat = torch.empty(300 * 19 + 1, dtype=torch.float64, device="cuda")
    view = flat[1:].view(300, 19)
    view.copy_(d.x)
    out = cf.hvp(fn, view, d.v, params=d.params)
    assert np.array_equal(out.cpu().numpy(), a, equal_nan=True)
    assert np.array_equal(dp.hessian(), d.hessian()[perm], equal_nan=True)
    Hflat = torch.empty(300 * 19 * 19 + 1, dtype=torch.float64, device="cuda")
    Hv = cf.hessian(fn, view, params=d.params, out=Hflat[1:].view(300, 19, 19))
    assert np.array_equal(Hv.cpu().numpy(), d.hessian(), equal_nan=True)


@pytest.mark.parametrize("prec", PRECS)
def test_fletcher_powell_several_points_per_cta_with_wide_rows(prec):
    """A batch that puts four points of n = 128 into a CTA (rows of A and B
    read past shared memory) and leaves a CTA with fewer."""
    d = Dev(W.make_batch(W.FLETCHER_POWELL, 128, 1215, seed=6), prec)
    assert hvp_err(d, d.hvp()).max() <= BOUND[prec]


@pytest.mark.parametrize("n", [12, 64, 128])
def test_ackley_fp32_off_the_16_byte_grid(n):
    """n a multiple of 4 with x, v and out 4 bytes off a 16-byte boundary, one
    at a time: the loads go element by element."""
    import torch

    d = Dev(W.make_batch(W.ACKLEY, n, 100, seed=n), cf.FP32_COMP)
    for which in range(3):
        t = [torch.empty(100 * n + 4, dtype=torch.float32, device="cuda") for _ in range(3)]
        x, v, out = [b[int(i == which):][:100 * n].view(100, n) for i, b in enumerate(t)]
        x.copy_(d.x)
        v.copy_(d.v)
        cf.hvp(W.ACKLEY, x, v, out=out)
        e = hvp_err(d, out.double().cpu().numpy())
        assert e.max() <= BOUND[cf.FP32_COMP], (which, e.max())


@pytest.mark.parametrize("fn", FNS)
@pytest.mark.parametrize("prec", PRECS)
def test_hessian_stores_whole_rows_or_not(fn, prec):
    """n a multiple of the values of a 16-byte store: an aligned output (a
    store's values together) and one that starts one element later (one by
    one) hold the same bits."""
    import torch

    for n in (4, 20, 64, 68):
        d = Dev(W.make_batch(fn, n, 37, seed=n), prec)
        flat = torch.empty(37 * n * n + 1, dtype=d.x.dtype, device="cuda")
        H = cf.hessian(fn, d.x, params=d.params, prec=prec, out=flat[1:].view(37, n, n))
        assert np.array_equal(H.double().cpu().numpy(), d.hessian())


@pytest.mark.parametrize("prec", PRECS)
def test_fletcher_powell_arguments_beyond_the_reduction(prec):
    """x on both sides of the range that sin and cos reduce themselves."""
    b = W.make_batch(W.FLETCHER_POWELL, 17, 60, seed=12)
    b.x[:30] *= 1e4
    b.x[30:] *= 1e7
    d = Dev(b, prec)
    assert hvp_err(d, d.hvp()).max() <= BOUND[prec]
    assert hessian_err(d, d.hessian()).max() <= BOUND[prec]


class _Uneven:
    """An uneven batch of the given functions and sizes and its plan (csize 0)."""

    def __init__(self, fns, ns, prec, seed=3):
        import torch

        self.fns, self.ns, self.prec = np.asarray(fns, np.int32), np.asarray(ns, np.int32), prec
        rng = np.random.Generator(np.random.PCG64(seed))
        self.fp = W.draw_fp_instance(rng, int(self.ns.max()))
        self.offs = np.concatenate([[0], np.cumsum(self.ns[:-1], dtype=np.int64)])
        x = np.concatenate([rng.uniform(*W.X_RANGE[int(f)], int(n)) for f, n in zip(fns, ns)])
        v = rng.uniform(-1, 1, int(self.ns.sum()))
        first, E, pos = {}, [], 0
        for n in sorted(set(self.ns.tolist())):
            E.append(W.fp_rhs(self.fp.A[:n, :n], self.fp.B[:n, :n], self.fp.alpha[:n]))
            first[n], pos = pos, pos + n
        self.eoffs = np.array([first[int(n)] for n in self.ns], np.int64)
        self.Epack = np.concatenate(E)
        dt = torch.float64 if prec == cf.FP64 else torch.float32
        self.x, self.v = torch.tensor(x, dtype=dt, device="cuda"), torch.tensor(v, dtype=dt, device="cuda")
        self.keep = [torch.tensor(t, device="cuda") for t in (self.fp.A, self.fp.B, self.Epack)]
        self.params = cf.fp_params(*self.keep)

    def reqs(self):
        return cf.requests(self.fns, self.ns, self.offs, self.eoffs)

    def run(self, csize=0):
        import torch

        plan = cf.RaggedPlan(self.reqs(), self.prec, csize)
        out = torch.full_like(self.x, 7.0)
        plan.run(self.x, self.v, out, self.params)
        torch.cuda.synchronize()
        first = out.double().cpu().numpy()
        plan.run(self.x, self.v, out, self.params)
        torch.cuda.synchronize()
        assert np.array_equal(first, out.double().cpu().numpy(), equal_nan=True)
        return first


@pytest.mark.parametrize("prec", PRECS)
def test_uneven_batch_tiles(prec):
    """Requests at the edges of the tiles: one variable, groups that end inside
    a tile, sizes that differ by more than a tile may mix, a few large
    Fletcher-Powell requests that are split over tiles; every request against
    the oracle, and a second run equal bit for bit."""
    import oracle
    from paper_2410_22575_gb300 import metrics

    F, R, A = W.FLETCHER_POWELL, W.ROSENBROCK, W.ACKLEY
    sizes = [1, 1, 2, 3, 5, 8, 9, 16, 17, 31, 32, 33, 64, 65, 100, 127, 128, 129, 200, 256, 257, 300, 511, 512]
    fns, ns = [], []
    for k, n in enumerate(sizes):
        for f in (F, R, A):
            fns += [f] * (1 + (k * 7 + f) % 3)
            ns += [n] * (1 + (k * 7 + f) % 3)
    order = np.random.Generator(np.random.PCG64(1)).permutation(len(ns))
    u = _Uneven(np.array(fns)[order], np.array(ns)[order], prec)
    got = u.run()
    xh, vh = u.x.double().cpu().numpy(), u.v.double().cpu().numpy()
    ref, hn = oracle.hvp_ragged(u.fns, u.ns, u.offs, u.eoffs, xh, vh, u.fp.A, u.fp.B, u.Epack, u.fp.A.shape[1])
    e = metrics.ragged_hvp_errors(got, ref, hn, vh, u.ns, u.offs)
    assert e.max() <= BOUND[prec], (e.max(), np.median(e))


@pytest.mark.parametrize("prec", PRECS)
def test_uneven_non_finite_requests_equal_the_dense_evaluation(prec):
    F, R, A = W.FLETCHER_POWELL, W.ROSENBROCK, W.ACKLEY
    fns = [F, R, A] * 8
    ns = [1] * 3 + [5] * 6 + [40] * 6 + [140] * 9
    u = _Uneven(fns, ns, prec)
    for k in range(0, 24, 2):
        t = u.x if k % 4 else u.v
        t[int(u.offs[k]) + u.ns[k] // 2] = (np.nan, np.inf, -np.inf)[k % 3]
    dense, got = u.run(8), u.run()
    fine = np.isfinite(dense)
    _same(got, dense, 4e-12 if prec == cf.FP64 else 4e-5, np.repeat(
        [np.max(np.abs(np.where(fine, dense, 0.0)[o:o + n]), initial=1.0) for o, n in zip(u.offs, u.ns)], u.ns)[fine])


# ------------------------------------------------------------------ user functions
@pytest.mark.parametrize("fn", [W.ROSENBROCK, W.ACKLEY, W.FLETCHER_POWELL, W.MIX])
@pytest.mark.parametrize("prec", PRECS)
def test_user_default_hvp(fn, prec):
    """The default product of a user function (one evaluation per chunk with d1
    seeded by v): chunk sizes that divide n, exceed it or leave a remainder, a
    point per CTA edge, and non-finite x and v, where it equals the symmetric
    method it replaces."""
    from test_gpu_user import SYM, Case, user_fn

    for c, n, batch in ((1, 5, 40), (8, 1, 300), (8, 8, 129), (8, 21, 50), (16, 7, 33), (16, 130, 3)):
        f, k = user_fn(fn, c, prec), Case(fn, n, batch, 40 + n, prec)
        out = f.hvp(k.x, k.v, k.params)
        e = k.hvp_err(out)
        assert e.max() <= BOUND[prec], (c, n, e.max())
        assert np.array_equal(out.cpu().numpy(), f.hvp(k.x, k.v, k.params).cpu().numpy())
    f, k = user_fn(fn, 8, prec), Case(fn, 21, 12, 7, prec)
    k.x[1, 4], k.x[2, 20], k.x[3, 0] = np.nan, np.inf, -np.inf
    k.v[4, 4], k.v[5, 20], k.v[6, 0] = np.nan, np.inf, -np.inf
    k.x[7, 3], k.v[7] = np.nan, 0.0
    got = f.hvp(k.x, k.v, k.params).double().cpu().numpy()
    dense = f.hvp(k.x, k.v, k.params, cfg=SYM).double().cpu().numpy()
    fine = np.isfinite(dense)
    scale = np.max(np.abs(np.where(fine, dense, 0.0)), axis=1, keepdims=True) * np.ones_like(dense)
    _same(got, dense, 4e-12 if prec == cf.FP64 else 4e-5, scale[fine])
