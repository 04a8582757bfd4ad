"""Sources that name the library's number type compile (no GPU needed: without
one, a source that compiles fails only at loading)."""
import pytest

import paper_2410_22575_gb300 as cf


@pytest.mark.parametrize("prec", [cf.FP64, cf.FP32_COMP])
def test_helper_on_the_number_type_compiles(prec):
    src = """template <class T, int C> __device__ chessfad::user::Num<T, C> cube(const chessfad::user::Num<T, C> &u)
    { return u * u * u; }
    template <class R, class X> R cubes(const X &x, int n, const double *p)
    { R f = 0.0; for (int k = 0; k < n; ++k) f += cube(x[k]) * x[0]; return f; }"""
    st, handle, log = cf.chessfad_user_fn_create(src, "cubes", 4, prec)
    assert st in (0, -10), (st, log)  # -10: compiled, no device to load it on
    if handle:
        cf.chessfad_user_fn_destroy(handle)


@pytest.mark.parametrize("prec", [cf.FP64, cf.FP32_COMP])
@pytest.mark.parametrize("csize", [1, 8])
def test_default_product_is_one_evaluation_per_chunk(prec, csize):
    """A source of the documented form, with every operator: both programs
    compile, and the log has nothing to say about the default product."""
    src = """template <class R, class X> R all_of_it(const X &x, int n, const double *p)
    {
        R f = 1.0;
        for (int k = 0; k < n; ++k) {
            R a = x[k], b = a;
            b += a; b -= 0.5 * a; b *= a; b /= 2.0 + a * a; b += 1.0; b -= 2.0; b *= 3.0; b /= 4.0;
            R c = a + b, d = a - b, e = a + 1.0, g = 1.0 + a, h = a - 1.0, i = 1.0 - a, j = a * 2.0;
            f += c * d + e / g - h * i + j / 3.0 + 1.0 / (4.0 + a * a) + (-b) + (+a);
            f += sin(a) + cos(a) + tan(0.1 * a) + tanh(a) + exp(-a) + log(3.0 + a * a) + sqrt(1.0 + a * a);
            f += pow(2.0 + a * a, 0.5) + abs(a) + fabs(b) + fmin(a, b) + fmax(a, b);
            if (a < b || a <= 0.0 || 1.0 > a || a >= b || a == b || a != 2.0) f += value(a) * b;
        }
        return f;
    }"""
    st, handle, log = cf.chessfad_user_fn_create(src, "all_of_it", csize, prec)
    assert st in (0, -10), (st, log)
    assert "symmetric" not in log and "error" not in log.split("loading failed")[0], log
    if handle:
        cf.chessfad_user_fn_destroy(handle)


def test_log_says_when_the_default_product_is_the_symmetric_one():
    src = """template <class T, int C> __device__ chessfad::user::Num<T, C> cube(const chessfad::user::Num<T, C> &u)
    { return u * u * u; }
    template <class R, class X> R cubes(const X &x, int n, const double *p) { return cube(x[0]); }"""
    st, handle, log = cf.chessfad_user_fn_create(src, "cubes", 4, cf.FP64)
    assert st in (0, -10) and "symmetric method" in log
    if handle:
        cf.chessfad_user_fn_destroy(handle)
