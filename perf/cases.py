"""What the speed of this library is measured on: Hessian-vector products and
Hessians through its public entry points, as a program that uses it calls them.

A case names the call (``kind``), the function, the sizes and the precision:

* ``hvp`` / ``hessian``: ``hvp(fn, x, v)`` / ``hessian(fn, x)`` on a [batch, n]
  device tensor, with the library's own choice of evaluation (``csize`` 0) or
  with a chunk size the caller asks for;
* ``host``: ``chessfad_hvp_host``, page-locked host tensors in and out;
* ``uneven``: a ``RaggedPlan`` of requests of different functions and sizes;
* ``user``: ``UserFunction.hvp`` of a function given as source text.

Inputs have the distributions of the library's own workloads: x uniform in
[-2, 2], [-5, 5] or [-pi, pi] by function, v in [-1, 1], Fletcher-Powell A, B
in [-100, 100] with E from a known zero.
"""
import functools
import math

import numpy as np
import torch

import paper_2410_22575_gb300 as cf

FNS = {"rosenbrock": cf.ROSENBROCK, "ackley": cf.ACKLEY, "fletcher_powell": cf.FLETCHER_POWELL}
X_MAX = {"rosenbrock": 2.0, "ackley": 5.0, "fletcher_powell": math.pi, "mix": 2.0}
DTYPE = {"f64": torch.float64, "f32": torch.float32}
PREC = {"f64": cf.FP64, "f32": cf.FP32_COMP}

# A function of the extended operator set, as a user writes it.
MIX = r"""
template <class R, class X>
R mix(const X &x, int n, const double *params)
{
    R f = 0.0;
    for (int k = 0; k + 1 < n; ++k) {
        R a = x[k], b = x[k + 1];
        R d = b - a;
        f += d * d / (1.0 + a * a) + abs(a) * b + tanh(a * b);
    }
    for (int k = 0; k < n; ++k) {
        R a = x[k];
        f += log(1.0 + a * a) + 0.1 * pow(2.0 + a * a, 1.5) + tan(0.3 * a);
    }
    return f;
}
"""


def _case(name, kind, fn, n, batch, dtype, csize=0):
    return {"name": name, "kind": kind, "fn": fn, "n": n, "batch": batch, "dtype": dtype, "csize": csize}


def listed():
    return [
        # a caller that needs one small batch now (an optimiser's inner step): latency
        _case("hvp_ackley_n8_f64_b32", "hvp", "ackley", 8, 32, "f64"),
        # the library's small stated workload, with the chunk size given
        _case("hvp_rosenbrock_n16_f64_chunk4", "hvp", "rosenbrock", 16, 4096, "f64", 4),
        # the headline workload, FP64
        _case("hvp_ackley_n64_f64", "hvp", "ackley", 64, 65536, "f64"),
        # half a million points (the batch of the method's own GPU experiments), compensated FP32
        _case("hvp_ackley_n64_f32_b512k", "hvp", "ackley", 64, 524288, "f32"),
        # the stated Fletcher-Powell workload, compensated FP32 with FP64 residuals
        _case("hvp_fletcher_powell_n32_f32", "hvp", "fletcher_powell", 32, 16384, "f32"),
        # an odd, larger Fletcher-Powell system in FP64
        _case("hvp_fletcher_powell_n75_f64", "hvp", "fletcher_powell", 75, 1000, "f64"),
        # the stated full-Hessian workload: many variables, output-heavy
        _case("hessian_rosenbrock_n256_f64", "hessian", "rosenbrock", 256, 1024, "f64"),
        # full Hessians of an odd number of variables, compensated FP32
        _case("hessian_ackley_n33_f32", "hessian", "ackley", 33, 20000, "f32"),
        # full Hessians of a dense coupled system, compensated FP32
        _case("hessian_fletcher_powell_n48_f32", "hessian", "fletcher_powell", 48, 4096, "f32"),
        # the uneven workload's mix of functions and sizes 2..512, a few thousand requests
        _case("uneven_n512_f32_r4000", "uneven", "all", 512, 4000, "f32"),
        # end to end from and to page-locked host memory
        _case("host_ackley_n64_f32", "host", "ackley", 64, 65536, "f32"),
        # a user-supplied function
        _case("user_mix_n64_f64", "user", "mix", 64, 4096, "f64", 8),
    ]


# A bound on a drawn case's cost, in operations of the dense chunked method
# (n^3 per point, n^4 for Fletcher-Powell), per precision.
_DENSE_OPS = {"f64": 1.5e11, "f32": 6e12}


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["hvp"] * 4 + ["hessian"] * 3 + ["uneven", "host", "user"])
    dtype = rng.choice(["f64", "f32"])
    if kind == "uneven":
        n = _log_uniform(rng, 32, 512 if dtype == "f32" else 160)
        most = 4000 if dtype == "f32" else 400
        return {"kind": kind, "fn": "all", "n": n, "batch": _log_uniform(rng, 20, most), "dtype": dtype, "csize": 0}
    fn = "mix" if kind == "user" else rng.choice(list(FNS))
    n = _log_uniform(rng, 2, 128 if kind == "user" else 512)
    dense = 8.0 * n ** 3 if fn != "fletcher_powell" else 4.0 * n ** 4
    if fn == "mix":
        dense *= 8.0
    most = min(524288, max(1, int(_DENSE_OPS[dtype] / dense)))
    if kind == "hessian":
        most = max(1, min(most, int(6e8 / (n * n * 8))))
    csize = 8 if kind == "user" else rng.choice([0] * 7 + [8])
    return {"kind": kind, "fn": fn, "n": n, "batch": _log_uniform(rng, min(16, most), most), "dtype": dtype,
            "csize": csize}


# ------------------------------------------------------------------ inputs
def _uniform(gen, shape, top):
    return (torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64) * 2 - 1) * top


def _system(gen, n):
    """Fletcher-Powell A, B and the alpha that is a zero of the residuals."""
    A = _uniform(gen, (n, n), 100.0)
    B = _uniform(gen, (n, n), 100.0)
    return A, B, _uniform(gen, (n,), math.pi)


def _rhs(A, B, alpha):
    return A @ torch.sin(alpha) + B @ torch.cos(alpha)


@functools.lru_cache(maxsize=None)
def _user_function(csize, dtype):
    return cf.UserFunction(MIX, "mix", csize, PREC[dtype])


def _inputs(case, seed):
    """x, v and the Fletcher-Powell data, on the GPU (the values the call sees)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, batch, fn = case["n"], case["batch"], case["fn"]
    fp = None
    if fn == "fletcher_powell":
        A, B, alpha = _system(gen, n)
        fp = (A, B, _rhs(A, B, alpha))
    x = _uniform(gen, (batch, n), X_MAX[fn]).to(DTYPE[case["dtype"]])
    v = _uniform(gen, (batch, n), 1.0).to(DTYPE[case["dtype"]])
    return x, v, fp


def _uneven_inputs(case, seed):
    """Requests of the three functions, sizes log-uniform in 2 .. n, packed.
    The table of requests belongs to the case, their values to the seed."""
    rng = np.random.Generator(np.random.PCG64(4))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    nreq, nmax = case["batch"], case["n"]
    fns = rng.integers(0, 3, nreq).astype(np.int32)
    ns = np.clip(np.rint(np.exp(rng.uniform(math.log(2), math.log(nmax), nreq))), 2, nmax).astype(np.int32)
    offs = np.concatenate([[0], np.cumsum(ns[:-1], dtype=np.int64)])
    A, B, alpha = _system(gen, nmax)
    sizes = sorted(set(ns[fns == cf.FLETCHER_POWELL].tolist())) or [1]
    E = torch.cat([_rhs(A[:k, :k], B[:k, :k], alpha[:k]) for k in sizes])
    first = dict(zip(sizes, np.concatenate([[0], np.cumsum(sizes[:-1])]).astype(np.int64).tolist()))
    eoffs = np.array([first[k] if f == cf.FLETCHER_POWELL else 0 for f, k in zip(fns.tolist(), ns.tolist())], np.int64)
    tops = np.array([X_MAX["rosenbrock"], X_MAX["ackley"], X_MAX["fletcher_powell"]])
    top = torch.as_tensor(np.repeat(tops[fns], ns), device="cuda")
    x = (_uniform(gen, (int(ns.sum()),), 1.0) * top).to(DTYPE[case["dtype"]])
    v = _uniform(gen, (int(ns.sum()),), 1.0).to(DTYPE[case["dtype"]])
    return fns, ns, offs, eoffs, x, v, A, B, E


def prepare(case, seed):
    kind, prec = case["kind"], PREC[case["dtype"]]
    state = {"case": case}
    if kind == "uneven":
        fns, ns, offs, eoffs, x, v, A, B, E = _uneven_inputs(case, seed)
        state.update(x=x, v=v, out=torch.empty_like(x), params=cf.fp_params(A, B, E), keep=(A, B, E))
        state["plan"] = cf.RaggedPlan(cf.requests(fns, ns, offs, eoffs), prec)
        return state
    x, v, fp = _inputs(case, seed)
    state.update(x=x, v=v, params=cf.fp_params(*fp) if fp else None, keep=fp)
    if kind == "user":
        state["f"] = _user_function(case["csize"], case["dtype"])
    elif kind == "host":
        state.update(xh=x.cpu().pin_memory(), vh=v.cpu().pin_memory(), dev=[torch.empty_like(x) for _ in range(3)])
        state["oh"] = torch.empty_like(state["xh"]).pin_memory()
    return state


# ------------------------------------------------------------------ one pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "hvp":
        return cf.hvp(FNS[case["fn"]], state["x"], state["v"], csize=case["csize"], params=state["params"])
    if kind == "hessian":
        return cf.hessian(FNS[case["fn"]], state["x"], csize=case["csize"], params=state["params"])
    if kind == "user":
        return state["f"].hvp(state["x"], state["v"])
    if kind == "uneven":
        return state["plan"].run(state["x"], state["v"], state["out"], state["params"])
    status = cf.chessfad_hvp_host(FNS[case["fn"]], case["n"], case["batch"], case["csize"], state["xh"], state["vh"],
                                  state["oh"], *state["dev"], state["params"], PREC[case["dtype"]])
    if status != cf.SUCCESS:
        raise cf.ChessfadError(status, "chessfad_hvp_host")
    return state["oh"]


# ------------------------------------------------------------------ work
def _hvp_flops(fn, n):
    """Operations one H v needs: the second derivatives' nonzero structure
    (tridiagonal; diagonal plus two rank-one parts; residual, J v and the
    transposed products), sin and cos at 20 operations each."""
    if fn == "rosenbrock":
        return 20.0 * n
    if fn == "ackley":
        return 60.0 * n
    if fn == "mix":
        return 250.0 * n
    return 16.0 * n * n + 60.0 * n


def work(case):
    size = 8 if case["dtype"] == "f64" else 4
    n, batch, fn = case["n"], case["batch"], case["fn"]
    if case["kind"] == "uneven":
        # means over n log-uniform in 2 .. nmax, a third of the requests each
        mean = (n - 2) / math.log(n / 2)
        square = (n * n - 4) / (2 * math.log(n / 2))
        flops = batch / 3 * (80.0 * mean + 16.0 * square + 60.0 * mean)
        return {"bytes": 3.0 * size * batch * mean + 16.0 * n * n, "flops": flops}
    system = 16.0 * n * n + 8.0 * n if fn == "fletcher_powell" else 0.0
    if case["kind"] != "hessian":
        return {"bytes": 3.0 * size * batch * n + system, "flops": batch * _hvp_flops(fn, n)}
    flops = {"rosenbrock": 15.0 * n, "ackley": 2.0 * n * n + 50.0 * n,
             "fletcher_powell": float(n) ** 3 + 10.0 * n * n}[fn]
    return {"bytes": float(size) * batch * (n + n * n) + system, "flops": batch * flops}


# ------------------------------------------------------------------ 64-bit values
def _value(fn, x, fp):
    """The sum of f over the rows of x (rows are independent, so derivatives
    of the sum are each row's own)."""
    if fn == "rosenbrock":
        a, b = x[:, :-1], x[:, 1:]
        return (100 * (b - a * a) ** 2 + (1 - a) ** 2).sum()
    if fn == "ackley":
        s, c = (x * x).mean(1), torch.cos(2 * math.pi * x).mean(1)
        return (-20 * torch.exp(-0.2 * torch.sqrt(s)) - torch.exp(c)).sum()
    if fn == "mix":
        a, b = x[:, :-1], x[:, 1:]
        f = ((b - a) ** 2 / (1 + a * a) + a.abs() * b + torch.tanh(a * b)).sum()
        return f + (torch.log(1 + x * x) + 0.1 * (2 + x * x) ** 1.5 + torch.tan(0.3 * x)).sum()
    A, B, E = fp
    r = E - torch.sin(x) @ A.T - torch.cos(x) @ B.T
    return (r * r).sum()


def _exact_hvp(fn, x, v, fp):
    x = x.double().detach().requires_grad_(True)
    if x.shape[1] == 1 and fn == "rosenbrock":
        return torch.zeros_like(x)
    g, = torch.autograd.grad(_value(fn, x, fp), x, create_graph=True)
    h, = torch.autograd.grad((g * v.double()).sum(), x)
    return h


def exact(case, seed):
    if case["kind"] == "uneven":
        fns, ns, offs, eoffs, x, v, A, B, E = _uneven_inputs(case, seed)
        out = torch.empty(x.shape, dtype=torch.float64, device="cuda")
        names = {i: name for name, i in FNS.items()}
        for f in sorted(set(fns.tolist())):
            for n in sorted(set(ns[fns == f].tolist())):
                sel = np.flatnonzero((fns == f) & (ns == n))
                at = torch.as_tensor(offs[sel][:, None] + np.arange(n), device="cuda")
                fp = None
                if f == cf.FLETCHER_POWELL:
                    e0 = int(eoffs[sel[0]])
                    fp = (A[:n, :n], B[:n, :n], E[e0:e0 + n])
                out[at] = _exact_hvp(names[f], x[at], v[at], fp)
        return out
    x, v, fp = _inputs(case, seed)
    if case["kind"] != "hessian":
        out = _exact_hvp(case["fn"], x, v, fp)
        return out.cpu() if case["kind"] == "host" else out
    rows = []
    for i in range(case["n"]):
        e = torch.zeros_like(x)
        e[:, i] = 1
        rows.append(_exact_hvp(case["fn"], x, e, fp))
    return torch.stack(rows, 1)
