// user_num.cuh -- the number type on which a user-supplied function is
// evaluated, and its operator set.  Compiled at run time (NVRTC) together
// with the user's source; see user_kernel.cuh and user.cu.
//
// Num<T, C> wraps one chunked hDual (hdual.cuh).  The user writes f once as a
// template on the number type (the library's premise, Sec. I and Sec. IV:
// f is overloaded on hDual so that one evaluation yields one chunk of one
// Hessian row).  The operators are the Fig. 1 rules and the unary chain rule
//   phi(u) = <phi(u), phi'(u) u_k, phi'(u) u_il + phi''(u) u_i u_l>
// with, per function:
//   sin    cos u, -sin u            cos   -sin u, -cos u
//   tan    1 + t^2, 2t(1 + t^2)     tanh  1 - t^2, -2t(1 - t^2)
//   exp    e^u, e^u                 log   1/u, -1/u^2
//   sqrt   1/(2 sqrt u), -1/(4 u^{3/2})
//   u^p    p u^{p-1}, p(p-1) u^{p-2} (p a real constant)
//   1/u    -1/u^2, 2/u^3            u / w = u * (1/w)
//   |u|    sign(u) u componentwise, sign(0) = +1
// Comparisons (Sec. IV lists them among the overloads) compare values;
// fmin / fmax return the operand the value comparison selects.
#pragma once

#include "hdual.cuh"

namespace chessfad {
namespace user {

// Scalar math by precision (distinct names, so the Num overloads below never
// hide the scalar ones inside this namespace).
__device__ __forceinline__ void m_sincos(float x, float &s, float &c) { sincosf(x, &s, &c); }
__device__ __forceinline__ void m_sincos(double x, double &s, double &c) { sincos(x, &s, &c); }
__device__ __forceinline__ float m_tan(float x) { return tanf(x); }
__device__ __forceinline__ double m_tan(double x) { return tan(x); }
__device__ __forceinline__ float m_tanh(float x) { return tanhf(x); }
__device__ __forceinline__ double m_tanh(double x) { return tanh(x); }
__device__ __forceinline__ float m_exp(float x) { return expf(x); }
__device__ __forceinline__ double m_exp(double x) { return exp(x); }
__device__ __forceinline__ float m_log(float x) { return logf(x); }
__device__ __forceinline__ double m_log(double x) { return log(x); }
__device__ __forceinline__ float m_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double m_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float m_pow(float x, float p) { return powf(x, p); }
__device__ __forceinline__ double m_pow(double x, double p) { return pow(x, p); }

// A derivative along the direction v (see DirVars): a sum over the variables.
// In FP32 it carries its rounding errors in e as Dot2 does (TwoProd, TwoSum), so
// that the sums over v are as accurate as the compensated row-times-v sums of
// the methods by rows; in FP64 it is one double.
template <typename T>
struct Dir;
template <>
struct Dir<double> {
    double s;
    __device__ __forceinline__ static Dir of(double x) { return Dir{x}; }
    __device__ __forceinline__ double value() const { return s; }
    __device__ __forceinline__ Dir operator+(const Dir &b) const { return Dir{s + b.s}; }
    __device__ __forceinline__ Dir operator-(const Dir &b) const { return Dir{s - b.s}; }
    __device__ __forceinline__ Dir operator-() const { return Dir{-s}; }
    __device__ __forceinline__ Dir operator*(double x) const { return Dir{x * s}; }
    __device__ __forceinline__ Dir operator/(double x) const { return Dir{s / x}; }
    // acc + x * this
    __device__ __forceinline__ Dir fma(double x, const Dir &acc) const { return Dir{__fma_rn(x, s, acc.s)}; }
};
template <>
struct Dir<float> {
    float s, e;
    __device__ __forceinline__ static Dir of(float x) { return Dir{x, 0.f}; }
    __device__ __forceinline__ float value() const { return __fadd_rn(s, e); }
    __device__ __forceinline__ Dir operator+(const Dir &b) const
    {
        Dir r;
        float t;
        two_sum(s, b.s, r.s, t);
        r.e = __fadd_rn(__fadd_rn(e, b.e), t);
        return r;
    }
    __device__ __forceinline__ Dir operator-(const Dir &b) const { return *this + (-b); }
    __device__ __forceinline__ Dir operator-() const { return Dir{-s, -e}; }
    __device__ __forceinline__ Dir operator*(float x) const
    {
        Dir r;
        float t;
        two_prod(x, s, r.s, t);
        r.e = __fmaf_rn(x, e, t);
        return r;
    }
    __device__ __forceinline__ Dir operator/(float x) const
    {
        const float q = s / x;
        return Dir{q, __fadd_rn(__fmaf_rn(-q, x, s), e) / x};
    }
    __device__ __forceinline__ Dir fma(float x, const Dir &acc) const
    {
        Dir r;
        float p, pe, t;
        two_prod(x, s, p, pe);
        two_sum(acc.s, p, r.s, t);
        r.e = __fadd_rn(acc.e, __fadd_rn(t, __fmaf_rn(x, e, pe)));
        return r;
    }
};

// Two of them, the operations packed (Dir<float>'s roundings: TwoProd's error is
// formed with the sign reversed, a - b as the exact fma(-1, b, a)).
struct Dir2 {
    float2 s, e;
    __device__ __forceinline__ static Dir2 both(const Dir<float> &d)
    {
        return Dir2{make_float2(d.s, d.s), make_float2(d.e, d.e)};
    }
    __device__ __forceinline__ static float2 sub(float2 a, float2 b)
    {
        return __ffma2_rn(make_float2(-1.f, -1.f), b, a);
    }
    __device__ __forceinline__ static void sum(float2 a, float2 b, float2 &s, float2 &t)
    {
        s = __fadd2_rn(a, b);
        const float2 bb = sub(s, a);
        t = __fadd2_rn(sub(a, sub(s, bb)), sub(b, bb));
    }
    __device__ __forceinline__ Dir2 operator+(const Dir2 &b) const
    {
        Dir2 r;
        float2 t;
        sum(s, b.s, r.s, t);
        r.e = __fadd2_rn(__fadd2_rn(e, b.e), t);
        return r;
    }
    __device__ __forceinline__ Dir2 operator*(float2 x) const
    {
        const float2 m = make_float2(-x.x, -x.y), p = __fmul2_rn(x, s), q = __ffma2_rn(m, s, p);
        return Dir2{p, __ffma2_rn(x, e, make_float2(-q.x, -q.y))};
    }
    __device__ __forceinline__ Dir2 fma(float2 x, const Dir2 &acc) const
    {
        const float2 m = make_float2(-x.x, -x.y), p = __fmul2_rn(x, s);
        const float2 q = __ffma2_rn(m, e, __ffma2_rn(m, s, p));
        Dir2 r;
        float2 t;
        sum(acc.s, p, r.s, t);
        r.e = __fadd2_rn(acc.e, sub(t, q));
        return r;
    }
};

// The components of a number of the directional evaluation: as HD, with d1 and
// h along v.
template <typename T, int C>
struct HDir {
    T v;
    Dir<T> d1;
    T g[C];
    Dir<T> h[C];
};

// f(l, ...) for every component l of h: f takes its arguments for one component,
// or in FP32 with an even C for two neighbours at a time.  at(): components l,
// l + 1 of h or g; all(): a scalar's or a derivative's value for both.
template <typename T>
struct One {
    template <int C>
    __device__ __forceinline__ static Dir<T> at(const Dir<T> (&h)[C], int l) { return h[l]; }
    template <int C>
    __device__ __forceinline__ static T at(const T (&g)[C], int l) { return g[l]; }
    __device__ __forceinline__ static T all(T x) { return x; }
    __device__ __forceinline__ static Dir<T> all(const Dir<T> &d) { return d; }
    template <int C>
    __device__ __forceinline__ static void put(Dir<T> (&h)[C], int l, const Dir<T> &d) { h[l] = d; }
};
struct Pair {
    template <int C>
    __device__ __forceinline__ static Dir2 at(const Dir<float> (&h)[C], int l)
    {
        return Dir2{make_float2(h[l].s, h[l + 1].s), make_float2(h[l].e, h[l + 1].e)};
    }
    template <int C>
    __device__ __forceinline__ static float2 at(const float (&g)[C], int l) { return make_float2(g[l], g[l + 1]); }
    __device__ __forceinline__ static float2 all(float x) { return make_float2(x, x); }
    __device__ __forceinline__ static Dir2 all(const Dir<float> &d) { return Dir2::both(d); }
    template <int C>
    __device__ __forceinline__ static void put(Dir<float> (&h)[C], int l, const Dir2 &d)
    {
        h[l] = Dir<float>{d.s.x, d.e.x};
        h[l + 1] = Dir<float>{d.s.y, d.e.y};
    }
};
template <typename T, int C, typename F>
__device__ __forceinline__ void components(Dir<T> (&h)[C], F &&f)
{
    if constexpr (sizeof(T) == 4 && C % 2 == 0) {
#pragma unroll
        for (int l = 0; l < C; l += 2) Pair::put(h, l, f(Pair(), l));
    } else {
#pragma unroll
        for (int l = 0; l < C; ++l) One<T>::put(h, l, f(One<T>(), l));
    }
}

// A: whether the number is one of the directional evaluation, which tracks
// activity.  In one evaluation a variable outside the chunk has zero g and h
// components, and so has everything computed from such variables alone; with A
// the zeros are neither stored nor multiplied (act is false), only the value
// and d1 are.  A skipped product would be an exact zero unless its other factor
// is Inf or NaN.  Such a factor makes d1 not finite, at the latest through the
// phi''(u) * 0 that the unary rule adds, and d1 stays so in whatever is computed
// from it; callers look at the result's d1.
template <typename T, int C, bool A = false>
struct Num;

// Members that both forms share.
#define CHESSFAD_USER_MEMBERS                                                                  \
    __device__ __forceinline__ T value() const { return a.v; }                                 \
    __device__ __forceinline__ Num &operator+=(const Num &w) { return *this = *this + w; }     \
    __device__ __forceinline__ Num &operator-=(const Num &w) { return *this = *this - w; }     \
    __device__ __forceinline__ Num &operator*=(const Num &w) { return *this = *this * w; }     \
    __device__ __forceinline__ Num &operator/=(const Num &w) { return *this = *this / w; }     \
    __device__ __forceinline__ Num &operator+=(double s) { a.v += T(s); return *this; }        \
    __device__ __forceinline__ Num &operator-=(double s) { a.v -= T(s); return *this; }        \
    __device__ __forceinline__ Num &operator*=(double s) { return *this = *this * s; }         \
    __device__ __forceinline__ Num &operator/=(double s) { return *this = *this / s; }
template <typename T, int C>
struct Num<T, C, false> {
    HD<T, C> a;

    __device__ __forceinline__ Num() : a(hzero<T, C>()) {}
    // A constant: value s, every derivative component zero.
    __device__ __forceinline__ Num(double s) : a(hzero<T, C>()) { a.v = T(s); }
    __device__ __forceinline__ explicit Num(const HD<T, C> &h) : a(h) {}
    CHESSFAD_USER_MEMBERS
};
template <typename T, int C>
struct Num<T, C, true> {
    HDir<T, C> a;
    bool act;

    __device__ __forceinline__ Num() : Num(0.0) {}
    __device__ __forceinline__ Num(double s) : act(false)
    {
        a.v = T(s);
        a.d1 = Dir<T>::of(T(0));
#pragma unroll
        for (int l = 0; l < C; ++l) {
            a.g[l] = T(0);
            a.h[l] = Dir<T>::of(T(0));
        }
    }
    CHESSFAD_USER_MEMBERS
};
#undef CHESSFAD_USER_MEMBERS

template <typename T, int C, bool A>
__device__ __forceinline__ T value(const Num<T, C, A> &u) { return u.a.v; }

// ---- arithmetic (Fig. 1)
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator+(const Num<T, C, A> &u, const Num<T, C, A> &w)
{
    if constexpr (!A) {
        return Num<T, C, A>(hadd(u.a, w.a));
    } else {
        Num<T, C, A> r = u;
        r.a.v = u.a.v + w.a.v;
        r.a.d1 = u.a.d1 + w.a.d1;
        if (w.act) {
            if (u.act) {
                vadd(u.a.g, w.a.g, r.a.g);
                components(r.a.h, [&](auto k, int l) { return k.at(u.a.h, l) + k.at(w.a.h, l); });
            } else {
#pragma unroll
                for (int l = 0; l < C; ++l) {
                    r.a.g[l] = w.a.g[l];
                    r.a.h[l] = w.a.h[l];
                }
            }
            r.act = true;
        }
        return r;
    }
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator-(const Num<T, C, A> &u, const Num<T, C, A> &w)
{
    if constexpr (!A) {
        return Num<T, C, A>(hsub(u.a, w.a));
    } else {
        Num<T, C, A> r = u + (-w);
        r.a.v = u.a.v - w.a.v;
        return r;
    }
}
// u * w with w inactive: the rule's terms without the zeros of w
template <typename T, int C>
__device__ __forceinline__ void hmul_by(const HDir<T, C> &u, const HDir<T, C> &w, HDir<T, C> &r)
{
    vmul(w.v, u.g, r.g);
    components(r.h, [&](auto k, int l) { return k.at(u.h, l).fma(k.all(w.v), k.all(w.d1) * k.at(u.g, l)); });
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator*(const Num<T, C, A> &u, const Num<T, C, A> &w)
{
    if constexpr (!A) {
        return Num<T, C, A>(hmul(u.a, w.a));
    } else {
        Num<T, C, A> r;
        if (u.act && w.act) {
            vmul(u.a.v, w.a.g, r.a.g);
            vfma(w.a.v, u.a.g, r.a.g);
            components(r.a.h, [&](auto k, int l) {
                auto h = k.at(w.a.h, l) * k.all(u.a.v);
                h = k.all(u.a.d1).fma(k.at(w.a.g, l), h);
                h = k.all(w.a.d1).fma(k.at(u.a.g, l), h);
                return k.at(u.a.h, l).fma(k.all(w.a.v), h);
            });
        } else if (u.act) {
            hmul_by(u.a, w.a, r.a);
        } else if (w.act) {
            hmul_by(w.a, u.a, r.a);
        }
        r.act = u.act || w.act;
        r.a.v = u.a.v * w.a.v;
        r.a.d1 = u.a.d1.fma(w.a.v, w.a.d1 * u.a.v);
        return r;
    }
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator-(const Num<T, C, A> &u)
{
    if constexpr (!A) {
        return Num<T, C, A>(rsub(T(0), u.a));
    } else {
        Num<T, C, A> r = u;
        r.a.v = T(0) - u.a.v;
        r.a.d1 = -u.a.d1;
        if (u.act) {
#pragma unroll
            for (int l = 0; l < C; ++l) {
                r.a.g[l] = -u.a.g[l];
                r.a.h[l] = -u.a.h[l];
            }
        }
        return r;
    }
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator+(const Num<T, C, A> &u) { return u; }

template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator+(const Num<T, C, A> &u, double s) { Num<T, C, A> r = u; r.a.v += T(s); return r; }
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator+(double s, const Num<T, C, A> &u) { Num<T, C, A> r = u; r.a.v = T(s) + r.a.v; return r; }
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator-(const Num<T, C, A> &u, double s) { Num<T, C, A> r = u; r.a.v -= T(s); return r; }
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator-(double s, const Num<T, C, A> &u)
{
    Num<T, C, A> r = -u;
    r.a.v = T(s) - u.a.v;
    return r;
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator*(const Num<T, C, A> &u, double s)
{
    if constexpr (!A) {
        return Num<T, C, A>(smul(T(s), u.a));
    } else {
        Num<T, C, A> r = u;
        r.a.v = T(s) * u.a.v;
        r.a.d1 = u.a.d1 * T(s);
        if (u.act) {
            vmul(T(s), u.a.g, r.a.g);
            components(r.a.h, [&](auto k, int l) { return k.at(u.a.h, l) * k.all(T(s)); });
        }
        return r;
    }
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator*(double s, const Num<T, C, A> &u) { return u * s; }

// phi(u) from phi, phi', phi'' at the value.
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> apply(const Num<T, C, A> &u, T phi, T d1, T d2)
{
    if constexpr (!A) {
        return Num<T, C, A>(unary(u.a, phi, d1, d2));
    } else {
        Num<T, C, A> r;
        r.a.v = phi;
        r.a.d1 = u.a.d1 * d1;
        if (u.act) {
            const Dir<T> q = u.a.d1 * d2;
            vmul(d1, u.a.g, r.a.g);
            components(r.a.h,
                       [&](auto k, int l) { return k.all(q).fma(k.at(u.a.g, l), k.at(u.a.h, l) * k.all(d1)); });
        } else {
            r.a.d1.s = fma_(d2, T(0), r.a.d1.s);
        }
        r.act = u.act;
        return r;
    }
}

template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> recip(const Num<T, C, A> &u)
{
    const T r = T(1) / u.a.v;
    return apply(u, r, -r * r, T(2) * r * r * r);
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator/(const Num<T, C, A> &u, const Num<T, C, A> &w) { return u * recip(w); }
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator/(double s, const Num<T, C, A> &w) { return s * recip(w); }
// u / s divides every component (correctly rounded per component).
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> operator/(const Num<T, C, A> &u, double s)
{
    const T d = T(s);
    Num<T, C, A> r = u;
    bool act = true;
    if constexpr (A) act = u.act;
    r.a.v = u.a.v / d;
    r.a.d1 = u.a.d1 / d;
    if (act) {
#pragma unroll
        for (int l = 0; l < C; ++l) {
            r.a.g[l] = u.a.g[l] / d;
            r.a.h[l] = u.a.h[l] / d;
        }
    }
    return r;
}

// ---- elementary functions
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> sin(const Num<T, C, A> &u)
{
    T s, c;
    m_sincos(u.a.v, s, c);
    return apply(u, s, c, -s);
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> cos(const Num<T, C, A> &u)
{
    T s, c;
    m_sincos(u.a.v, s, c);
    return apply(u, c, -s, -c);
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> tan(const Num<T, C, A> &u)
{
    const T t = m_tan(u.a.v), d = T(1) + t * t;
    return apply(u, t, d, T(2) * t * d);
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> tanh(const Num<T, C, A> &u)
{
    const T t = m_tanh(u.a.v), d = T(1) - t * t;
    return apply(u, t, d, T(-2) * t * d);
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> exp(const Num<T, C, A> &u)
{
    const T e = m_exp(u.a.v);
    return apply(u, e, e, e);
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> log(const Num<T, C, A> &u)
{
    const T r = T(1) / u.a.v;
    return apply(u, m_log(u.a.v), r, -r * r);
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> sqrt(const Num<T, C, A> &u)
{
    const T s = m_sqrt(u.a.v), d = T(0.5) / s;
    return apply(u, s, d, -d / (T(2) * u.a.v));
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> pow(const Num<T, C, A> &u, double p)
{
    // Three powers, so that each has pow()'s own accuracy (u^0 is 1 and the
    // derivative of u^1 is 1).  A number outside the chunk uses phi'' only to
    // notice that it is not finite; where u^(p-2) = u^(p-1) / u and its factor
    // are far inside the range, that power is left out (the extended-operator
    // test function, FP64, n = 64, 4096 points: 1.67 ms with three powers
    // everywhere, 1.30 so).
    const T q = T(p), x = u.a.v, big = sizeof(T) == 8 ? T(1e75) : T(1e9);
    const T w0 = m_pow(x, q), w1 = m_pow(x, q - T(1));
    bool needed = !(x > T(1) / big && x < big && w1 < big && q < big && q > -big);
    if constexpr (A) needed |= u.act;
    else needed = true;
    const T w = needed ? m_pow(x, q - T(2)) : T(0);
    return apply(u, w0, q * w1, q * (q - T(1)) * w);
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> abs(const Num<T, C, A> &u)
{
    return u.a.v < T(0) ? -u : u;
}
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> fabs(const Num<T, C, A> &u) { return abs(u); }

// ---- comparisons on values
#define CHESSFAD_USER_CMP(op)                                                                               \
    template <typename T, int C, bool A>                                                                           \
    __device__ __forceinline__ bool operator op(const Num<T, C, A> &u, const Num<T, C, A> &w) { return u.a.v op w.a.v; } \
    template <typename T, int C, bool A>                                                                           \
    __device__ __forceinline__ bool operator op(const Num<T, C, A> &u, double s) { return u.a.v op T(s); }    \
    template <typename T, int C, bool A>                                                                           \
    __device__ __forceinline__ bool operator op(double s, const Num<T, C, A> &u) { return T(s) op u.a.v; }
CHESSFAD_USER_CMP(<)
CHESSFAD_USER_CMP(<=)
CHESSFAD_USER_CMP(>)
CHESSFAD_USER_CMP(>=)
CHESSFAD_USER_CMP(==)
CHESSFAD_USER_CMP(!=)
#undef CHESSFAD_USER_CMP

template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> fmin(const Num<T, C, A> &u, const Num<T, C, A> &w) { return w.a.v < u.a.v ? w : u; }
template <typename T, int C, bool A>
__device__ __forceinline__ Num<T, C, A> fmax(const Num<T, C, A> &u, const Num<T, C, A> &w) { return w.a.v > u.a.v ? w : u; }

// The variables x_0 .. x_{n-1} of one evaluation: x[k] is the CHUNK-INIT
// seed of variable k (Alg. 4) for Hessian row i and the chunk starting at
// cstart, generated on the fly; its zeros are opaque (dense arithmetic).
template <typename T, int C>
struct Vars {
    const T *x;
    int i, cstart;
    SeedK<T> z;
    __device__ __forceinline__ Num<T, C> operator[](int k) const { return Num<T, C>(seed<T, C>(x[k], k, i, cstart, z)); }
};

// The same for a product H v in one evaluation per chunk: d1 is seeded by the
// direction v instead of the unit vector of a row, so the result's h
// components are (H v)_(cstart + l).
template <typename T, int C>
struct DirVars {
    const T *x, *v;
    int stride, cstart;
    SeedK<T> z;
    __device__ __forceinline__ Num<T, C, true> operator[](int k) const
    {
        // x, v: this point's variables, `stride` elements apart
        Num<T, C, true> y;
        y.a.v = x[k * stride];
        y.a.d1 = Dir<T>::of(v[k * stride]);
        const int d = k - cstart;
        y.act = d >= 0 && d < C;
        if (y.act) {
#pragma unroll
            for (int l = 0; l < C; ++l) {
                y.a.g[l] = (d == l) ? z.one : z.z;
                y.a.h[l] = Dir<T>::of(z.z);
            }
        }
        return y;
    }
};

}  // namespace user
}  // namespace chessfad
