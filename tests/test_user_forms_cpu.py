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
