// structured.cuh -- Hessian-vector products and Hessians of the built-in
// functions by the hDual rules applied to the components that the seeding
// makes nonzero.
//
// The dense sweeps (sweep.cuh) evaluate f once per (row i, chunk) on hDuals
// in which every variable but x_i and the chunk's has a zero derivative part;
// almost all of their arithmetic is products with those seed zeros.  Here the
// rules of hdual.cuh are applied to the nonzero components only, and for a
// product H v the seed of d1 is the direction v itself: with d1 seeded by v_k
// instead of [k == i], the h component of variable l is (H v)_l directly, so
// one pass over a point replaces its n rows.
//
//   Rosenbrock       row l holds three entries (two neighbouring terms);
//                    their products with v are summed as the dense row is.
//   Ackley           the two sums under sqrt and exp carry
//                    d1 = sum_k x_k v_k and sum_k phi'(x_k) v_k; the tail's
//                    unary rules then give each (H v)_l from g and h of its
//                    own variable.
//   Fletcher-Powell  residual r_m carries its FP64 value and
//                    d1_m = -(J v)_m; the squares' rule needs sum_m d1_m g_ml
//                    and sum_m r_m h_ml, four transposed products with A, B.
//
// A product with a seed zero is an exact zero unless its other factor is Inf
// or NaN, and there the dense method returns NaN.  Points whose result is not
// finite are therefore evaluated again entry by entry with the dense method's
// propagation (the *_dense_* functions below), so non-finite inputs and
// overflow give what the dense sweeps give.
#pragma once

#include <cuda_runtime.h>
#include <math_constants.h>

#include "fp64_sincos.cuh"
#include "hdual.cuh"
#include "sweep.cuh"

namespace chessfad {

// Tests and conversions of FP64 values on 32-bit words: a comparison or an
// absolute value (also a mask of the sign bit of the whole 64-bit word, which
// the compiler makes one of) is an FP64 instruction.
__device__ __forceinline__ bool not_finite(float x) { return (__float_as_uint(x) & 0x7f800000u) == 0x7f800000u; }
__device__ __forceinline__ bool not_finite(double x)
{
    return ((unsigned)__double2hiint(x) & 0x7ff00000u) == 0x7ff00000u;
}

__device__ __forceinline__ float nan_of(float) { return CUDART_NAN_F; }
__device__ __forceinline__ double nan_of(double) { return CUDART_NAN; }

// float -> double through the integer pipe: the conversion instruction runs at
// the FP64 pipe's rate, 1/64 of FP32's.  Exact for normal floats; zeros and
// subnormals become 0 (the callers add squares and cosines: such a square,
// below 2^-252, is nothing in S/n as a float), Inf and NaN a finite value
// (callers take points with those another way).
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x)
{
    const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
    const unsigned hi = (b & 0x80000000u) | ((m >> 3) + 0x38000000u);
    const bool zero = m < 0x00800000u;
    return __hiloint2double(zero ? 0 : (int)hi, zero ? 0 : (int)(b << 29));
}

// double -> float, round to nearest even, through the integer pipe.  A result
// that would be a subnormal float becomes NaN: its point is then evaluated again
// by the dense propagation, which converts with the instruction.  (The
// instruction here, for such values alone, took the 4000-request uneven batch
// from 256 to 287 us.)  Below half the smallest subnormal: 0.
template <typename T>
__device__ __forceinline__ T narrow(double x);
template <>
__device__ __forceinline__ double narrow<double>(double x) { return x; }
template <>
__device__ __forceinline__ float narrow<float>(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x), h = hi & 0x7fffffffu;
    unsigned r = __funnelshift_l(lo, h, 3);  // exponent and 23 bits; 29 bits of lo are dropped
    r += (((lo & 0x1fffffffu) + 0x0fffffffu + (r & 1u)) >> 29) - (896u << 23);
    if (h < (897u << 20)) r = h < (873u << 20) ? 0u : 0x7fffffffu;
    if (h >= (1151u << 20)) r = h > 0x7ff00000u || (h == 0x7ff00000u && lo) ? 0x7fffffffu : 0x7f800000u;
    return __uint_as_float(r | (hi & 0x80000000u));
}

// The row-times-v sum of the dense sweeps: Dot2 in compensated FP32, FMAs in
// FP64.
template <typename T>
struct RowSum;
template <>
struct RowSum<float> {
    CSum s{0.f, 0.f};
    __device__ __forceinline__ void add(float a, float b) { cdot_add(s, a, b); }
    __device__ __forceinline__ float value() const { return csum_value(s); }
    __device__ __forceinline__ void merge_xor(int off)
    {
        CSum o;
        o.s = __shfl_xor_sync(0xffffffffu, s.s, off);
        o.e = __shfl_xor_sync(0xffffffffu, s.e, off);
        s = csum_merge(s, o);
    }
};
template <>
struct RowSum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double a, double b) { s = __fma_rn(a, b, s); }
    __device__ __forceinline__ double value() const { return s; }
    __device__ __forceinline__ void merge_xor(int off) { s += __shfl_xor_sync(0xffffffffu, s, off); }
};

// Row s of a point evaluated densely: sum_j entry(s, j) v_j over every j.
// wide: the dense HVP of this size adds its rows in FP64 (SymStage) instead
// of as a Dot2.
template <typename T, typename IO, typename F>
__device__ __forceinline__ T dense_row(const IO *v, int n, int s, bool wide, F &&entry)
{
    if (IsComp<T>::value && wide) {
        double d = 0.0;
        for (int j = 0; j < n; ++j) d = fma((double)entry(s, j), (double)v[j], d);
        return (T)d;
    }
    RowSum<T> d;
    for (int j = 0; j < n; ++j) d.add(entry(s, j), (T)v[j]);
    return d.value();
}

// ------------------------------------------------------------------ Rosenbrock
// Row l of the Hessian from the terms k = l - 1 (as its y_{k+1}: d.d1 = d.g =
// 1) and k = l (as its y_k: d.d1 = d.g = -2 x_l, d.h = -2), each square by the
// unary rule; the rounding is the dense sweep's.
template <typename T>
struct RosRow {
    T lo, diag, up;  // entries (l, l-1), (l, l), (l, l+1)
};
template <typename T>
__device__ __forceinline__ RosRow<T> ros_row(T xm, T x0, T xp, int l, int n)
{
    RosRow<T> r;
    r.lo = T(0);
    r.diag = T(0);
    r.up = T(0);
    if (l > 0) {
        r.lo = T(200) * (T(-2) * xm);
        r.diag = T(200);
    }
    if (l < n - 1) {
        const T g = T(-2) * x0;
        const T dv = fma_(T(-1), x0 * x0, xp);
        r.up = T(200) * g;
        r.diag = fma_(r.up, g, r.diag);
        r.diag = fma_(T(200) * dv, T(-2), r.diag);
        r.diag = r.diag + T(2);
    }
    return r;
}

// What non-finite terms do to the dense entries.  A term whose x_k is not
// finite multiplies seed zeros of every component: every entry is NaN.  A
// term whose residual 200 d overflows (x_k finite) multiplies only second
// derivatives, zero except at (k, k): every other entry is NaN.
struct RosBad {
    int count, at;  // residual-overflow terms, the last one's index
    bool all;
};
template <typename T, typename IO>
__device__ __forceinline__ RosBad ros_bad(const IO *x, int n)
{
    RosBad b{0, -1, false};
    for (int k = 0; k + 1 < n; ++k) {
        const T x0 = (T)x[k], dv = fma_(T(-1), x0 * x0, (T)x[k + 1]);
        if (not_finite(x0)) b.all = true;
        else if (not_finite(T(200) * dv)) {
            ++b.count;
            b.at = k;
        }
    }
    return b;
}
template <typename T, typename IO>
__device__ __forceinline__ T ros_dense_entry(const IO *x, int n, const RosBad &b, int i, int j)
{
    if (b.all || (b.count > 0 && !(b.count == 1 && i == j && b.at == i))) return nan_of(T(0));
    if (i - j > 1 || j - i > 1) return T(0);
    const RosRow<T> r = ros_row<T>(i > 0 ? (T)x[i - 1] : T(0), (T)x[i], i + 1 < n ? (T)x[i + 1] : T(0), i, n);
    const T v = j < i ? r.lo : j == i ? r.diag : r.up;
    // an infinite term leaves a NaN in the TwoSum of compensated FP32
    return IsComp<T>::value && not_finite(v) ? nan_of(T(0)) : v;
}
template <typename T, typename IO>
__device__ __noinline__ void ros_dense_hvp(const IO *x, const IO *v, IO *out, int n, int t, int G, bool wide)
{
    const RosBad b = ros_bad<T>(x, n);
    for (int s = t; s < n; s += G)
        out[s] = (IO)dense_row<T>(v, n, s, wide, [&](int i, int j) { return ros_dense_entry<T>(x, n, b, i, j); });
}

// H v of one point by the G lanes t = 0 .. G-1 of an aligned group of its
// warp (every lane of the warp calls it; idle groups pass active = false).
template <typename T, typename IO>
__device__ __forceinline__ void ros_point(const IO *__restrict__ x, const IO *__restrict__ v, IO *__restrict__ out,
                                          int n, int t, int G, bool active, bool wide)
{
    bool bad = false;
    if (active) {
#pragma unroll 4
        for (int l = t; l < n; l += G) {
            const bool lo = l > 0, hi = l < n - 1;
            const T xm = lo ? (T)x[l - 1] : T(0), x0 = (T)x[l], xp = hi ? (T)x[l + 1] : T(0);
            const T vm = lo ? (T)v[l - 1] : T(0), v0 = (T)v[l], vp = hi ? (T)v[l + 1] : T(0);
            const RosRow<T> r = ros_row<T>(xm, x0, xp, l, n);
            RowSum<T> d;
            d.add(r.lo, vm);
            d.add(r.diag, v0);
            d.add(r.up, vp);
            const T o = d.value();
            bad |= not_finite(o);
            out[l] = (IO)o;
        }
    }
    // a not finite x, v or residual makes its own row's product not finite
    const unsigned votes = __ballot_sync(0xffffffffu, bad);
    const unsigned mask = (G == 32 ? 0xffffffffu : ((1u << G) - 1u)) << ((threadIdx.x & 31) - t);
    if (votes & mask) {
        __syncwarp(mask);
        ros_dense_hvp<T>(x, v, out, n, t, G, wide);
    }
}

// ------------------------------------------------------------------ Ackley
// sin and cos of 2 pi x; the FP64 form keeps its coefficients in registers.
template <typename T>
struct Turn;
template <>
struct Turn<float> {
    __device__ __forceinline__ void operator()(float x, float &s, float &c) const { sincospif(2.0f * x, &s, &c); }
};
template <>
struct Turn<double> {
    SinCosK k = sincos_k(1);
    __device__ __forceinline__ void operator()(double x, double &s, double &c) const { sincos_turn(k, x, s, c); }
};

// The tail's derivative factors of one point, from S = sum x^2 and
// C = sum cos 2 pi x (both FP64): r = sqrt(S/n) as a function of S/2,
// -20 exp(-0.2 r) as a function of r, -exp(C/n) as a function of C.
template <typename T>
struct AckTail {
    T r1, r2;  // r', r''
    T p1, p2;  // of -20 exp(-0.2 r)
    T q1, q2;  // of -exp(C/n), times -4 pi^2 and 4 pi^2: the factors that
               // cos 2 pi x's phi'' = -4 pi^2 cos and phi' = -2 pi sin (twice)
               // leave when C's components are taken as plain cos and sin
    // -20 exp(-0.2 r) as a function of S/2: the two unary rules composed
    __device__ __forceinline__ T f1() const { return p1 * r1; }
    __device__ __forceinline__ T f2() const { return fma_(p1, r2, (p2 * r1) * r1); }
};
// The constant factors of n variables: 1/n, 1/n^2, 4 pi^2/n and -4 pi^2/n^2,
// in compensated FP32 as unevaluated pairs (the rounded constant alone would
// put the same error into every point).  One per launch.
struct AckConst {
    double inv_n, k[4];
    float hi[4], lo[4];
};
__host__ __device__ inline AckConst ack_const(int n)
{
    AckConst c;
    const double four_pi_sq = 39.478417604357434475337963999504604541254797628963;
    c.inv_n = 1.0 / n;
    c.k[0] = c.inv_n;
    c.k[1] = 1.0 / ((double)n * n);
    c.k[2] = four_pi_sq * c.k[0];
    c.k[3] = -four_pi_sq * c.k[1];
    for (int i = 0; i < 4; ++i) {
        c.hi[i] = (float)c.k[i];
        c.lo[i] = (float)(c.k[i] - (double)c.hi[i]);
    }
    return c;
}

// The scalar functions in FP64, or, for compensated FP32, in FP32 from the
// correctly rounded FP64 sums.  pair: the thread's neighbour (lane xor 1)
// holds the same point and the two share the exponentials; every lane of the
// warp calls it then.
__device__ __forceinline__ AckTail<double> ack_tail(double S, double C, const AckConst &n, bool pair, double)
{
    AckTail<double> k;
    const double a0 = S * n.inv_n, sq = sqrt(a0), w = 1.0 / (sq * a0);
    double e1, e2;
    if (pair) {
        const bool odd = threadIdx.x & 1;
        const double e = exp(odd ? C * n.inv_n : -0.2 * sq), o = __shfl_xor_sync(0xffffffffu, e, 1);
        e1 = odd ? o : e;
        e2 = odd ? e : o;
    } else {
        e1 = exp(-0.2 * sq);
        e2 = exp(C * n.inv_n);
    }
    k.r1 = (n.k[0] * a0) * w;
    k.r2 = -n.k[1] * w;
    k.p1 = 4.0 * e1;
    k.p2 = -0.8 * e1;
    k.q1 = n.k[2] * e2;
    k.q2 = n.k[3] * e2;
    return k;
}
// In compensated FP32, from a0 = S/n and c = C/n.
__device__ __forceinline__ AckTail<float> ack_tail_f(float a0, float c, const AckConst &n)
{
    AckTail<float> k;
    const float sq = sqrtf(a0);
    const float e1 = expf(-0.2f * sq), e2 = expf(c);
    const float d1 = 1.0f / sq, d2 = -1.0f / (sq * a0);
    auto times = [&](int i, float y) { return __fmaf_rn(n.hi[i], y, n.lo[i] * y); };
    k.r1 = times(0, d1);
    k.r2 = times(1, d2);
    k.p1 = 4.0f * e1;
    k.p2 = -0.8f * e1;
    k.q1 = times(2, e2);
    k.q2 = times(3, e2);
    return k;
}
__device__ __forceinline__ AckTail<float> ack_tail(double S, double C, const AckConst &n, bool, float)
{
    return ack_tail_f(narrow<float>(S * n.inv_n), narrow<float>(C * n.inv_n), n);
}

// One variable's h component of the whole tail: S/2 carries (d1 = sd, g = x,
// h = sh), C carries (d1 = cd, g = cg, h = ch) in the units of q1, q2.  As the
// dense sweep composes it, rule by rule:
template <typename T>
__device__ __forceinline__ T ack_tail_h(const AckTail<T> &k, T sd, T x, T sh, T cd, T cg, T ch)
{
    HD<T, 1> a, b;
    a.v = b.v = T(0);
    a.d1 = sd;
    a.g[0] = x;
    a.h[0] = sh;
    b.d1 = cd;
    b.g[0] = cg;
    b.h[0] = ch;
    const HD<T, 1> r = unary(a, T(0), k.r1, k.r2);
    HD<T, 1> f = unary(r, T(0), k.p1, k.p2);
    add_unary<false>(f, b, T(0), k.q1, k.q2);
    return f.h[0];
}

// A point evaluated as the dense sweeps propagate non-finite values: a not
// finite x_k multiplies seed zeros in S of every component.
template <typename T, typename IO>
struct AckDense {
    const IO *x;
    bool poison;
    AckTail<T> k;
    __device__ __forceinline__ AckDense(const IO *x_, int n) : x(x_), poison(false)
    {
        const Turn<T> turn;
        double S = 0.0, C = 0.0;
        for (int j = 0; j < n; ++j) {
            T s, c;
            const T xj = (T)x[j];
            turn(xj, s, c);
            poison |= not_finite(xj);
            S = fma((double)xj, (double)xj, S);
            C += (double)c;
        }
        k = ack_tail(S, C, ack_const(n), false, T(0));
        // the sqrt rule's factors at any S, as the dense prologue forms them
        const T a0 = (T)(S / n), sq = sqrt(a0), k2 = T(2) * T(1.0 / n);
        k.r1 = k2 * (T(0.5) / sq);
        k.r2 = (k2 * k2) * (T(-0.25) / (sq * a0));
    }
    __device__ __forceinline__ T entry(int i, int j) const
    {
        if (poison) return nan_of(T(0));
        const Turn<T> turn;
        T si, ci, sj, cj;
        turn((T)x[i], si, ci);
        turn((T)x[j], sj, cj);
        return ack_tail_h<T>(k, (T)x[i], (T)x[j], i == j ? T(1) : T(0), si, sj, i == j ? cj : T(0));
    }
};
template <typename T, typename IO>
__device__ __noinline__ void ack_dense_hvp(const IO *x, const IO *v, IO *out, int n, int t, int G, bool wide)
{
    const AckDense<T, IO> d(x, n);
    for (int s = t; s < n; s += G)
        out[s] = (IO)dense_row<T>(v, n, s, wide, [&](int i, int j) { return d.entry(i, j); });
}

// The four sums of one point: S = sum x^2, C = sum cos 2 pi x and the
// direction's sum x v and sum sin(2 pi x) v, over a lane's variables, then
// over the G lanes of its group.
template <typename T>
struct AckSums;
template <>
struct AckSums<double> {
    double S = 0.0, C = 0.0, X = 0.0, Y = 0.0;
    __device__ __forceinline__ void add(double x, double v, double s, double c)
    {
        S = fma(x, x, S);
        C += c;
        X = fma(x, v, X);
        Y = fma(s, v, Y);
    }
    __device__ __forceinline__ void merge(int G)
    {
        for (int off = G >> 1; off > 0; off >>= 1) {
            S += __shfl_xor_sync(0xffffffffu, S, off);
            C += __shfl_xor_sync(0xffffffffu, C, off);
            X += __shfl_xor_sync(0xffffffffu, X, off);
            Y += __shfl_xor_sync(0xffffffffu, Y, off);
        }
    }
    __device__ __forceinline__ AckTail<double> tail(const AckConst &n, bool pair) const
    {
        return ack_tail(S, C, n, pair, 0.0);
    }
    __device__ __forceinline__ double x() const { return X; }
    __device__ __forceinline__ double y() const { return Y; }
    __device__ __forceinline__ bool small() const { return false; }
};
// Compensated FP32: Dot2 and Sum2 (the error term catches the rounding of
// every product and addition, so a sum is as accurate as one formed in twice
// FP32's precision), the sums two by two in packed instructions: (S, X) of
// x * (x, v), (Y, C) of (s, c) * (v, 1).  FP64 sums of the same values took
// 60 % of the kernel's time, on a pipe with 1/64 of the FP32 rate, for bits
// that the rounding of S/n and C/n to FP32 discards.
template <>
struct AckSums<float> {
    float2 p, pe, q, qe;  // (S, X), (Y, C) and their errors
    __device__ __forceinline__ AckSums()
    {
        p = pe = q = qe = make_float2(0.f, 0.f);
    }
    // (s, e) += a * b by TwoProd and TwoSum
    __device__ __forceinline__ static void dot2(float2 &s, float2 &e, float2 a, float2 b)
    {
        const float2 m1 = make_float2(-1.f, -1.f);
        const float2 w = __fmul2_rn(a, b), we = __ffma2_rn(a, b, make_float2(-w.x, -w.y));
        const float2 t = __fadd2_rn(s, w), bb = __ffma2_rn(m1, s, t);
        const float2 u = __ffma2_rn(m1, __ffma2_rn(m1, bb, t), s), z = __ffma2_rn(m1, bb, w);
        e = __fadd2_rn(e, __fadd2_rn(__fadd2_rn(u, z), we));
        s = t;
    }
    __device__ __forceinline__ void add(float x, float v, float s, float c)
    {
        dot2(p, pe, make_float2(x, x), make_float2(x, v));
        dot2(q, qe, make_float2(s, c), make_float2(v, 1.0f));
    }
    __device__ __forceinline__ static void merge1(float &s, float &e, int off)
    {
        CSum o;
        o.s = __shfl_xor_sync(0xffffffffu, s, off);
        o.e = __shfl_xor_sync(0xffffffffu, e, off);
        o = csum_merge(CSum{s, e}, o);
        s = o.s;
        e = o.e;
    }
    // From 4 lanes on, each lane keeps two of the four sums at the first
    // distance and one at the second, and fetches the others at the end: 3 +
    // log2(G / 4) merges instead of 4 log2(G).
    __device__ __forceinline__ void merge(int G)
    {
        if (G < 4) {
            for (int off = G >> 1; off > 0; off >>= 1) {
                merge1(p.x, pe.x, off);
                merge1(p.y, pe.y, off);
                merge1(q.x, qe.x, off);
                merge1(q.y, qe.y, off);
            }
            return;
        }
        const int lane = threadIdx.x & 31, a = G >> 1, b = G >> 2;
        const bool ha = lane & a, hb = lane & b;
        CSum k0 = half(ha, CSum{p.x, pe.x}, CSum{q.x, qe.x}, a), k1 = half(ha, CSum{p.y, pe.y}, CSum{q.y, qe.y}, a);
        k0 = half(hb, k0, k1, b);
        for (int off = b >> 1; off > 0; off >>= 1) merge1(k0.s, k0.e, off);
        const int at = lane & ~(G - 1);
        p.x = __shfl_sync(0xffffffffu, k0.s, at);
        pe.x = __shfl_sync(0xffffffffu, k0.e, at);
        p.y = __shfl_sync(0xffffffffu, k0.s, at + b);
        pe.y = __shfl_sync(0xffffffffu, k0.e, at + b);
        q.x = __shfl_sync(0xffffffffu, k0.s, at + a);
        qe.x = __shfl_sync(0xffffffffu, k0.e, at + a);
        q.y = __shfl_sync(0xffffffffu, k0.s, at + a + b);
        qe.y = __shfl_sync(0xffffffffu, k0.e, at + a + b);
    }
    // x (high: y) merged with the partner's
    __device__ __forceinline__ static CSum half(bool high, const CSum &x, const CSum &y, int off)
    {
        const CSum keep = high ? y : x, give = high ? x : y;
        CSum o;
        o.s = __shfl_xor_sync(0xffffffffu, give.s, off);
        o.e = __shfl_xor_sync(0xffffffffu, give.e, off);
        return csum_merge(keep, o);
    }
    // (s + e) / n, rounded once but for the last bits of the small terms
    __device__ __forceinline__ static float over_n(float s, float e, const AckConst &n)
    {
        return __fmaf_rn(n.hi[0], s, __fmaf_rn(n.hi[0], e, n.lo[0] * s));
    }
    __device__ __forceinline__ AckTail<float> tail(const AckConst &n, bool) const
    {
        return ack_tail_f(over_n(p.x, pe.x, n), over_n(q.y, qe.y, n), n);
    }
    __device__ __forceinline__ float x() const { return __fadd_rn(p.y, pe.y); }
    __device__ __forceinline__ float y() const { return __fadd_rn(q.x, qe.x); }
    // squares whose TwoProd error underflows: the point goes the dense way
    // (FP64 sums)
    __device__ __forceinline__ bool small() const { return p.x < 1e-30f; }
};

// A load the compiler may not replace by the value of an earlier one.
__device__ __forceinline__ double load_again(const double *p)
{
    double r;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(r) : "l"(p));
    return r;
}
__device__ __forceinline__ float load_again(const float *p)
{
    float r;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(r) : "l"(p));
    return r;
}

// H v of one point by the G lanes of an aligned group of its warp, EPL
// variables per lane, n <= G EPL: variable t + G j, or, kVec (float, n a
// multiple of 4, 16-byte aligned x, v, out), four neighbours at a time.
template <typename T, typename IO, int EPL, bool kVec = false>
__device__ __forceinline__ void ack_point(const IO *__restrict__ x, const IO *__restrict__ v, IO *__restrict__ out,
                                          int n, int t, int G, bool active, bool wide,
                                          const AckConst &nc)
{
    const int m = active ? n : 0;
    const Turn<T> turn;
    constexpr int V = kVec ? 4 : 1;
    auto var = [&](int j) { return V == 1 ? t + G * j : 4 * (t + G * (j / 4)) + j % 4; };
    // FP64 with many variables per lane: x and v are read again (from L1) for
    // the tail instead of held in 4 EPL registers, so that twice the warps
    // keep the FP64 pipe filled.
    constexpr bool kReload = sizeof(T) == 8 && EPL >= 8;
    constexpr int kHeld = kReload ? 1 : EPL;
    T xs[kHeld], vs[kHeld], sn[EPL], cs[EPL];
    AckSums<T> sum;
    if constexpr (kVec) {
#pragma unroll
        for (int j = 0; j < EPL; j += 4) {
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            if (var(j) < m) {
                a = *reinterpret_cast<const float4 *>(x + var(j));
                b = *reinterpret_cast<const float4 *>(v + var(j));
            }
            xs[j] = a.x, xs[j + 1] = a.y, xs[j + 2] = a.z, xs[j + 3] = a.w;
            vs[j] = b.x, vs[j + 1] = b.y, vs[j + 2] = b.z, vs[j + 3] = b.w;
        }
    } else if constexpr (!kReload) {
#pragma unroll
        for (int j = 0; j < EPL; ++j) {
            const int k = var(j);
            xs[j] = T(0);
            vs[j] = T(0);
            if (k < m) {
                xs[j] = (T)x[k];
                vs[j] = (T)v[k];
            }
        }
    }
#pragma unroll
    for (int j = 0; j < EPL; ++j) {
        if (V * G * (j / V) < n) {  // uniform in the group
            const bool on = var(j) < m;
            if constexpr (kReload) {
                xs[0] = on ? (T)x[t + G * j] : T(0);
                vs[0] = on ? (T)v[t + G * j] : T(0);
            }
            const T xj = xs[kReload ? 0 : j], vj = vs[kReload ? 0 : j];
            turn(xj, sn[j], cs[j]);
            if (on) sum.add(xj, vj, sn[j], cs[j]);
        }
    }
    sum.merge(G);
    const AckTail<T> k = sum.tail(nc, G > 1);
    bool bad = active && sum.small();
    if (active) {
        // f1 h + (f2 d1) g of S/2 plus q1 h + (q2 d1) g of C
        const T f1 = k.f1(), fx = k.f2() * sum.x(), qs = k.q2 * sum.y();
        T o4[V];
#pragma unroll
        for (int j = 0; j < EPL; ++j) {
            if (var(j) < n) {
                T xj, vj;
                if constexpr (kReload) {
                    xj = (T)load_again(x + t + G * j);
                    vj = (T)load_again(v + t + G * j);
                } else {
                    xj = xs[j];
                    vj = vs[j];
                }
                T o = fma_(fx, xj, f1 * vj);
                o = fma_(qs, sn[j], o);
                o = fma_(k.q1, cs[j] * vj, o);
                bad |= not_finite(o);
                o4[j % V] = o;
                if constexpr (!kVec) out[var(j)] = (IO)o;
                else if (j % 4 == 3)
                    *reinterpret_cast<float4 *>(out + var(j - 3)) = make_float4(o4[0], o4[1], o4[2], o4[3]);
            }
        }
    }
    // a not finite x makes S or C, a not finite v its own row, not finite
    const unsigned votes = __ballot_sync(0xffffffffu, bad);
    const unsigned mask = (G == 32 ? 0xffffffffu : ((1u << G) - 1u)) << ((threadIdx.x & 31) - t);
    if (votes & mask) {
        __syncwarp(mask);
        ack_dense_hvp<T>(x, v, out, n, t, G, wide);
    }
}

// ------------------------------------------------------------------ Fletcher-Powell
// A CTA of kFpThreads holds up to kFpPairs (point, variable) pairs, points
// q < P of sizes n_q packed one after the other (pair base_q + j).
//   pass 1  r_m = E_m - sum_j (A_mj sin x_j + B_mj cos x_j) in FP64 and
//           d1_m = -sum_j (A_mj cos x_j - B_mj sin x_j) v_j, for the rows m of
//           an A/B tile in shared memory, L lanes per (point, row);
//   pass 2  sum_m A_ml d1_m, B_ml d1_m, A_ml r_m, B_ml r_m of every pair, kept
//           in registers across the tiles, kFpNpt pairs per thread.
// In compensated FP32 only the residual is FP64 (2 of the 8 FMAs of an (m, j)
// pair), and the FP64 pipe is the bound all the same; the other sums add
// blocks of plain FP32 FMAs with TwoSum.
constexpr int kFpThreads = 256;
constexpr int kFpNpt = 2;
constexpr int kFpPairs = kFpThreads * kFpNpt;
constexpr int kFpMaxPts = 128;

struct FpShape {
    int nmax;   // largest n of the tile's points
    int mt;     // rows of A, B per shared-memory tile
    int bufs;   // tile buffers: 2 when the rows take several tiles; 0: wide rows
    int pairs;  // (point, variable) pairs the shared arrays hold
    int lanes;  // lanes per (point, row) in pass 1, a power of two <= 32; wide
                // rows: (point, row) items per warp, 2 or 4
};

// Two values read and multiplied together: (A, B) of one (m, j), (sin, cos)
// of one variable.
template <typename T>
struct alignas(2 * sizeof(T)) Two {
    T x, y;
};

// Shared-memory layout (bytes) of a CTA.  The A/B tile holds (A, B) pairs in
// FP64 and, in compensated FP32, once more rounded, for the FP32 sums.
template <typename T>
struct FpSmem {
    size_t z, t, rd, ab, fab, q, base, n, xoff, eoff, total;
};
// Row stride of the tiles in pairs: odd, so lanes on different rows (pass 1)
// hit different banks.
__host__ __device__ inline int fp_stride(int nmax) { return nmax | 1; }

template <typename T>
__host__ __device__ inline FpSmem<T> fp_smem(const FpShape &sh)
{
    FpSmem<T> s{};
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off = align_up(off + bytes, 16);
        return at;
    };
    const size_t tile = (size_t)sh.bufs * sh.mt * fp_stride(sh.nmax), np = (size_t)sh.pairs;
    s.xoff = take(kFpMaxPts * sizeof(long long));
    s.eoff = take(kFpMaxPts * sizeof(long long));
    s.z = take(np * sizeof(Two<double>));
    s.t = take(np * sizeof(Two<T>));
    s.rd = take(np * sizeof(Two<T>));
    s.ab = take(tile * sizeof(Two<double>));
    s.fab = s.ab;
    if (sizeof(T) == 4) s.fab = take((sh.bufs ? tile : (size_t)sh.mt * fp_stride(sh.nmax)) * sizeof(Two<T>));
    s.n = take(kFpMaxPts * sizeof(int));
    s.base = take((kFpMaxPts + 1) * sizeof(int));
    s.q = take(np);
    s.total = off;
    return s;
}

// N pairs of sums over products of a Two with a Two or with a scalar: pass 1's
// one pair per (point, row), pass 2's per (point, variable).
template <typename T, int N>
struct FpSums;
template <int N>
struct FpSums<double, N> {
    double s[2 * N];
    __device__ __forceinline__ void init()
    {
#pragma unroll
        for (int i = 0; i < 2 * N; ++i) s[i] = 0.0;
    }
    __device__ __forceinline__ void add(int i, const Two<double> &a, double x, double y)
    {
        s[2 * i] = __fma_rn(a.x, x, s[2 * i]);
        s[2 * i + 1] = __fma_rn(a.y, y, s[2 * i + 1]);
    }
    __device__ __forceinline__ void flush() {}
    __device__ __forceinline__ double value(int i) const { return s[i]; }
    __device__ __forceinline__ double wide(int i) const { return s[i]; }
    __device__ __forceinline__ RowSum<double> both() const
    {
        RowSum<double> r;
        r.s = s[0] + s[1];
        return r;
    }
};
// Compensated FP32: packed FMAs into block partials p, which flush() adds into
// the pairs (s, e) with TwoSum (a - b as the exact fma(-1, b, a)).
template <int N>
struct FpSums<float, N> {
    float2 s[N], e[N], p[N];
    __device__ __forceinline__ void init()
    {
#pragma unroll
        for (int i = 0; i < N; ++i) s[i] = e[i] = p[i] = make_float2(0.f, 0.f);
    }
    __device__ __forceinline__ void add(int i, const Two<float> &a, float x, float y)
    {
        p[i] = __ffma2_rn(make_float2(a.x, a.y), make_float2(x, y), p[i]);
    }
    __device__ __forceinline__ void flush()
    {
        const float2 m1 = make_float2(-1.f, -1.f);
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const float2 t = __fadd2_rn(s[i], p[i]), bb = __ffma2_rn(m1, s[i], t);
            const float2 x = __ffma2_rn(m1, __ffma2_rn(m1, bb, t), s[i]), y = __ffma2_rn(m1, bb, p[i]);
            e[i] = __fadd2_rn(e[i], __fadd2_rn(x, y));
            s[i] = t;
            p[i] = make_float2(0.f, 0.f);
        }
    }
    __device__ __forceinline__ CSum sum(int i) const
    {
        return i & 1 ? CSum{s[i / 2].y, e[i / 2].y} : CSum{s[i / 2].x, e[i / 2].x};
    }
    __device__ __forceinline__ float value(int i) const { return csum_value(sum(i)); }
    __device__ __forceinline__ double wide(int i) const { return (double)sum(i).s + (double)sum(i).e; }
    __device__ __forceinline__ RowSum<float> both() const
    {
        RowSum<float> r;
        r.s = csum_merge(sum(0), sum(1));
        return r;
    }
};
// (a block partial is kSumBlock plain FP32 FMAs per sum)

struct FpArgs {
    const double *A, *B, *E;
    int ld;
};

// One tile of points.  The caller has filled, in shared memory, n[q], base[q]
// (base[P] = the pair count), xoff[q] and eoff[q], and synchronised.
// Afterwards sums[i] holds the four pass-2 sums of pair tid + i kFpThreads
// over the rows m0 <= m < m1.
// kDir: with the direction v (products H v); without it only r_m and the two
// sums over it (the Hessian's diagonal part).
template <typename T, typename IO, bool kDir>
struct FpTile {
    static constexpr int NS = kDir ? 2 : 1;
    const FpArgs a;
    const IO *x, *v;
    unsigned char *smem;
    const FpShape sh;
    const FpSmem<T> L;
    const int P, npairs;
    Two<double> *z, *ab;  // (sin, cos); (A, B)
    Two<T> *t, *rd, *fab;  // v (cos, -sin); (r, d1); (A, B)
    unsigned char *qs;
    int *ns, *base;
    long long *xoff, *eoff;

    __device__ __forceinline__ FpTile(const FpArgs &a_, const IO *x_, const IO *v_, unsigned char *sm,
                                      const FpShape &s, int P_, int npairs_)
        : a(a_), x(x_), v(v_), smem(sm), sh(s), L(fp_smem<T>(s)), P(P_), npairs(npairs_)
    {
        z = reinterpret_cast<Two<double> *>(sm + L.z);
        ab = reinterpret_cast<Two<double> *>(sm + L.ab);
        t = reinterpret_cast<Two<T> *>(sm + L.t);
        rd = reinterpret_cast<Two<T> *>(sm + L.rd);
        fab = reinterpret_cast<Two<T> *>(sm + L.fab);
        qs = sm + L.q;
        ns = reinterpret_cast<int *>(sm + L.n);
        base = reinterpret_cast<int *>(sm + L.base);
        xoff = reinterpret_cast<long long *>(sm + L.xoff);
        eoff = reinterpret_cast<long long *>(sm + L.eoff);
    }

    // sin, cos (FP64) and their products with v of every pair
    __device__ __forceinline__ void stage()
    {
        const SinCosK k = sincos_k(0);
        for (int u = threadIdx.x; u < npairs; u += kFpThreads) {
            int lo = 0, hi = P - 1;  // the pair's point: base[lo] <= u < base[lo + 1]
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (base[mid] <= u) lo = mid;
                else hi = mid - 1;
            }
            qs[u] = (unsigned char)lo;
            const long long o = xoff[lo] + (u - base[lo]);
            double s, c;
            sincos_rad(k, (double)x[o], s, c);
            z[u] = Two<double>{s, c};
            if constexpr (kDir) {
                const T vv = (T)v[o];
                t[u] = Two<T>{narrow<T>(c) * vv, -(narrow<T>(s) * vv)};
            }
        }
    }

    // Start the copy of rows [mb, mend) of A and B into a tile buffer (8-byte
    // cp.async: any leading dimension and base alignment).
    __device__ __forceinline__ void load_tile(int buf, int mb, int mend)
    {
        const int w = fp_stride(sh.nmax), cnt = (mend - mb) * sh.nmax, o = buf * sh.mt * w;
        for (int e = threadIdx.x; e < cnt; e += kFpThreads) {
            const int mm = e / sh.nmax, j = e - mm * sh.nmax;
            const size_t g = (size_t)(mb + mm) * a.ld + j;
            const unsigned d = (unsigned)__cvta_generic_to_shared(ab + o + mm * w + j);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(a.A + g));
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d + 8u), "l"(a.B + g));
        }
        asm volatile("cp.async.commit_group;");
    }
    // Round what this thread copied, once it has arrived.
    __device__ __forceinline__ void round_tile(int buf, int mb, int mend)
    {
        if constexpr (sizeof(T) == 4) {
            const int w = fp_stride(sh.nmax), cnt = (mend - mb) * sh.nmax, o = buf * sh.mt * w;
            for (int e = threadIdx.x; e < cnt; e += kFpThreads) {
                const int mm = e / sh.nmax, d = o + mm * w + e - mm * sh.nmax;
                fab[d] = Two<T>{narrow<T>(ab[d].x), narrow<T>(ab[d].y)};
            }
        }
    }

    // pass 1 over the rows [mb, mend) in a buffer; every lane of a warp runs
    // the same number of items (the shuffles)
    __device__ __forceinline__ void residuals(int buf, int mb, int mend)
    {
        const int w = fp_stride(sh.nmax), mt = mend - mb, lanes = sh.lanes;
        const int lane = threadIdx.x & (lanes - 1), items = P * mt, groups = kFpThreads / lanes;
        const int iters = (items + groups - 1) / groups;
        for (int it = 0; it < iters; ++it) {
            const int idx = threadIdx.x / lanes + it * groups;
            int q = 0, mm = 0, n = 0;
            if (idx < items) {
                q = idx / mt;
                mm = idx - q * mt;
                if (mb + mm < ns[q]) n = ns[q];
            }
            const int z0 = base[q], row = (buf * sh.mt + mm) * w;
            double s = 0.0, s2 = 0.0;  // two chains: the FP64 latency is several issue slots
            FpSums<T, 1> d;
            d.init();
            auto term = [&](int j) {
                const Two<double> g = ab[row + j], zz = z[z0 + j];
                s = fma(g.x, zz.x, s);
                s2 = fma(g.y, zz.y, s2);
                if constexpr (kDir) {
                    const Two<T> tt = t[z0 + j];
                    d.add(0, fab[row + j], tt.x, tt.y);
                }
            };
            int j = lane;
            for (; j + (kSumBlock - 1) * lanes < n; j += kSumBlock * lanes) {
#pragma unroll
                for (int i = 0; i < kSumBlock; ++i) term(j + i * lanes);
                if constexpr (kDir) d.flush();
            }
            for (; j < n; j += lanes) term(j);
            if constexpr (kDir) d.flush();
            s += s2;
            RowSum<T> d1 = d.both();
            for (int off = lanes >> 1; off > 0; off >>= 1) {
                s += __shfl_xor_sync(0xffffffffu, s, off);
                if constexpr (kDir) d1.merge_xor(off);
            }
            if (n > 0 && lane == 0)
                rd[z0 + mb + mm] = Two<T>{narrow<T>(a.E[eoff[q] + mb + mm] - s), kDir ? -d1.value() : T(0)};
        }
    }

    // pass 2 over the rows in a buffer
    __device__ __forceinline__ void transposed(int buf, int mb, int mend, FpSums<T, NS> (&sums)[kFpNpt])
    {
        const int w = fp_stride(sh.nmax);
#pragma unroll
        for (int i = 0; i < kFpNpt; ++i) {
            const int u = threadIdx.x + i * kFpThreads;
            if (u >= npairs) break;
            const int q = qs[u], z0 = base[q], end = min(mend, ns[q]);
            const Two<T> *g = fab + buf * sh.mt * w + (u - z0), *f = rd + z0;
            auto term = [&](int m) {
                const Two<T> gg = g[(m - mb) * w], ff = f[m];
                sums[i].add(0, gg, ff.x, ff.x);
                if constexpr (kDir) sums[i].add(1, gg, ff.y, ff.y);
            };
            int m = mb;
            for (; m + kSumBlock <= end; m += kSumBlock) {
#pragma unroll
                for (int k = 0; k < kSumBlock; ++k) term(m + k);
                sums[i].flush();
            }
            for (; m < end; ++m) term(m);
            sums[i].flush();
        }
    }

    // Wide rows (few points per CTA): A and B come straight from L2.  A warp
    // takes S (point, row) items at a time, its lanes the columns; after a
    // barrier the threads add the items' rows to their columns, in compensated
    // FP32 from the rounded rows that pass 1 left in shared memory.
    template <int S>
    __device__ __forceinline__ void run_wide(int m0, int m1, FpSums<T, NS> (&sums)[kFpNpt])
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, w = fp_stride(sh.nmax), chunk = sh.mt;
        for (int mb = m0; mb < m1; mb += chunk) {
            const int mend = min(mb + chunk, m1), items = (mend - mb) * P;
            __syncthreads();  // sin and cos are staged; the last chunk's rows are read
            double s[S], s2[S];
            FpSums<T, 1> d[S];
            int z0[S], n[S], row[S];
            const double *Ar[S], *Br[S];
            bool put[S];
#pragma unroll
            for (int v = 0; v < S; ++v) {
                // a row's points on neighbouring slots; its first point leaves
                // the rounded row (the points are ordered by size)
                const int idx = warp * S + v, q = idx < items ? idx % P : 0, m = mb + (idx < items ? idx / P : 0);
                z0[v] = base[q];
                n[v] = idx < items && m < ns[q] ? ns[q] : 0;
                put[v] = sizeof(T) == 4 && idx < items && q == 0;
                row[v] = (m - mb) * w;
                Ar[v] = a.A + (size_t)m * a.ld;
                Br[v] = a.B + (size_t)m * a.ld;
                s[v] = s2[v] = 0.0;
                d[v].init();
            }
            int blk = 0;
            // 64 columns at a time, the next ones' loads under this one's sums
            double av[2][S], bv[2][S], an[2][S], bn[2][S];
            auto fetch = [&](int j0, double (&x)[2][S], double (&y)[2][S]) {
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int v = 0; v < S; ++v) {
                        const int j = j0 + 32 * h;
                        x[h][v] = y[h][v] = 0.0;
                        if (j < (put[v] ? sh.nmax : n[v])) {
                            x[h][v] = __ldg(Ar[v] + j);
                            y[h][v] = __ldg(Br[v] + j);
                        }
                    }
            };
            constexpr bool kAhead = S == 2;  // four items have loads enough, and registers for no more
            if (kAhead) fetch(lane, an, bn);
            for (int j0 = lane; j0 < sh.nmax; j0 += 64) {
                if constexpr (kAhead) {
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int v = 0; v < S; ++v) {
                            av[h][v] = an[h][v];
                            bv[h][v] = bn[h][v];
                        }
                    fetch(j0 + 64, an, bn);
                } else {
                    fetch(j0, av, bv);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int v = 0; v < S; ++v) {
                        const int j = j0 + 32 * h;
                        const Two<T> g{narrow<T>(av[h][v]), narrow<T>(bv[h][v])};
                        if (put[v] && j < sh.nmax) fab[row[v] + j] = g;
                        if (j < n[v]) {
                            const Two<double> zz = z[z0[v] + j];
                            s[v] = fma(av[h][v], zz.x, s[v]);
                            s2[v] = fma(bv[h][v], zz.y, s2[v]);
                            if constexpr (kDir) {
                                const Two<T> tt = t[z0[v] + j];
                                d[v].add(0, g, tt.x, tt.y);
                            }
                        }
                    }
                blk += 2;
                if (kDir && blk == kSumBlock) {
                    blk = 0;
#pragma unroll
                    for (int v = 0; v < S; ++v) d[v].flush();
                }
            }
            // Across the lanes: halve the slots a lane holds at distances 16
            // and, with four, 8 (6 additions for four sums, 5 for two).
            RowSum<T> e[S];
#pragma unroll
            for (int v = 0; v < S; ++v) {
                s[v] += s2[v];
                if constexpr (kDir) d[v].flush();
                e[v] = d[v].both();
            }
            const bool h16 = lane & 16, h8 = lane & 8;
#pragma unroll
            for (int v = 0; v < S / 2; ++v) {
                fold(s[v], s[v + S / 2], h16, 16);
                if constexpr (kDir) fold_row(e[v], e[v + S / 2], h16, 16);
            }
            if constexpr (S == 4) {
                fold(s[0], s[1], h8, 8);
                if constexpr (kDir) fold_row(e[0], e[1], h8, 8);
            }
            for (int off = S == 4 ? 4 : 8; off > 0; off >>= 1) {
                s[0] += __shfl_xor_sync(0xffffffffu, s[0], off);
                if constexpr (kDir) e[0].merge_xor(off);
            }
            const int idx = warp * S + (S == 4 ? (h16 ? 2 : 0) + (h8 ? 1 : 0) : (h16 ? 1 : 0));
            if ((lane & (S == 4 ? 7 : 15)) == 0 && idx < items) {
                const int q = idx % P, m = mb + idx / P;
                if (m < ns[q])
                    rd[base[q] + m] = Two<T>{narrow<T>(a.E[eoff[q] + m] - s[0]), kDir ? -e[0].value() : T(0)};
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kFpNpt; ++i) {
                const int u = threadIdx.x + i * kFpThreads;
                if (u >= npairs) break;
                const int q = qs[u], l = u - base[q], end = min(mend, ns[q]);
                const Two<T> *f = rd + base[q], *g = fab + l;
                const double *Al = a.A + l, *Bl = a.B + l;
                auto term = [&](int m) {
                    const Two<T> ff = f[m];
                    Two<T> gg;
                    if constexpr (sizeof(T) == 4) {
                        gg = g[(m - mb) * w];
                    } else {
                        gg.x = __ldg(Al + (size_t)m * a.ld);
                        gg.y = __ldg(Bl + (size_t)m * a.ld);
                    }
                    sums[i].add(0, gg, ff.x, ff.x);
                    if constexpr (kDir) sums[i].add(1, gg, ff.y, ff.y);
                };
                int m = mb;
                for (; m + kSumBlock <= end; m += kSumBlock) {
#pragma unroll
                    for (int k = 0; k < kSumBlock; ++k) term(m + k);
                    sums[i].flush();
                }
                for (; m < end; ++m) term(m);
                sums[i].flush();
            }
        }
        __syncthreads();
    }
    // lanes with `high` keep b, the others a, each adding its partner's part
    __device__ __forceinline__ static void fold(double &x, double &y, bool high, int off)
    {
        const double keep = high ? y : x, give = high ? x : y;
        x = keep + __shfl_xor_sync(0xffffffffu, give, off);
    }
    __device__ __forceinline__ static void fold_row(RowSum<double> &x, RowSum<double> &y, bool high, int off)
    {
        fold(x.s, y.s, high, off);
    }
    __device__ __forceinline__ static void fold_row(RowSum<float> &x, RowSum<float> &y, bool high, int off)
    {
        const CSum keep = high ? y.s : x.s, give = high ? x.s : y.s;
        CSum o;
        o.s = __shfl_xor_sync(0xffffffffu, give.s, off);
        o.e = __shfl_xor_sync(0xffffffffu, give.e, off);
        x.s = csum_merge(keep, o);
    }

    // Rows m0 <= m < m1.  The next tile's copy runs under this tile's passes.
    template <bool kWide>
    __device__ __forceinline__ void run(int m0, int m1, FpSums<T, NS> (&sums)[kFpNpt])
    {
#pragma unroll
        for (int i = 0; i < kFpNpt; ++i) sums[i].init();
        if constexpr (kWide) {
            stage();
            if (sh.lanes == 4) run_wide<4>(m0, m1, sums);
            else run_wide<2>(m0, m1, sums);
            return;
        }
        load_tile(0, m0, min(m0 + sh.mt, m1));
        stage();
        int buf = 0;
        for (int mb = m0; mb < m1; mb += sh.mt, buf ^= 1) {
            const int mend = min(mb + sh.mt, m1);
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            round_tile(buf, mb, mend);
            __syncthreads();  // the tile has arrived, and the other buffer is read no more
            if (mend < m1) load_tile(buf ^ 1, mend, min(mend + sh.mt, m1));
            residuals(buf, mb, mend);
            __syncthreads();
            transposed(buf, mb, mend, sums);
        }
        __syncthreads();
    }

    // (H v)_l = 2 sum_m [d1_m g_ml + r_m h_ml], g_ml = -(A_ml cos - B_ml sin),
    // h_ml = (A_ml sin + B_ml cos) v_l
    __device__ __forceinline__ T combine(int u, T ar, T br, T ad, T bd) const
    {
        const T s = narrow<T>(z[u].x), c = narrow<T>(z[u].y), vv = (T)v[xoff[qs[u]] + (u - base[qs[u]])];
        RowSum<T> o;
        o.add(-c, ad);
        o.add(s, bd);
        o.add(s * vv, ar);
        o.add(c * vv, br);
        return T(2) * o.value();
    }
    // the diagonal's second-derivative part, 2 sum_m r_m (A_ml sin + B_ml cos)
    __device__ __forceinline__ T curvature(int u, const FpSums<T, 1> &sum) const
    {
        RowSum<T> o;
        o.add(narrow<T>(z[u].x), sum.value(0));
        o.add(narrow<T>(z[u].y), sum.value(1));
        return T(2) * o.value();
    }
};

// One point for the dense propagation: sin, cos (FP64) and the residuals of
// every variable.  An x, A or B that is not finite multiplies seed zeros in
// some residual of every component (poison).
template <typename T>
struct FpDense {
    const double *A, *B;
    int ld, n;
    const Two<double> *z;
    const Two<T> *r;  // .x
    bool poison;
    __device__ __forceinline__ T entry(int i, int j) const
    {
        if (poison) return nan_of(T(0));
        const T si = (T)z[i].x, ci = (T)z[i].y, sj = (T)z[j].x, cj = (T)z[j].y;
        const T hs = i == j ? -sj : T(0), hc = i == j ? -cj : T(0);
        TermSum<T, 1, IsComp<T>::value> acc;
        acc.init();
        for (int m = 0; m < n; ++m) {
            const double *Ar = A + (size_t)m * ld, *Br = B + (size_t)m * ld;
            HD<T, 1> t;
            t.v = r[m].x;
            t.d1 = -fma_((T)Br[i], -si, (T)Ar[i] * ci);
            t.g[0] = -fma_((T)Br[j], -sj, (T)Ar[j] * cj);
            t.h[0] = -fma_((T)Br[j], hc, (T)Ar[j] * hs);
            acc.add_sq(t);
        }
        return acc.value().h[0];
    }
};

// Whether x or the leading n x n block of A or B holds a value that is not
// finite in T; every thread of the CTA calls it.
template <typename T, typename IO>
__device__ __forceinline__ bool fp_poison(const FpArgs &a, const IO *x, int n)
{
    bool p = false;
    for (int l = threadIdx.x; l < n; l += blockDim.x) p |= not_finite((T)x[l]);
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        const size_t at = (size_t)(e / n) * a.ld + e % n;
        p |= not_finite((T)a.A[at]) || not_finite((T)a.B[at]);
    }
    return __syncthreads_or(p);
}

// r_m of every m from the staged sin and cos; every thread calls it.
template <typename T>
__device__ __forceinline__ void fp_residuals(const FpArgs &a, const double *E, int n, const Two<double> *z, Two<T> *r)
{
    for (int m = threadIdx.x; m < n; m += blockDim.x) {
        double s = 0.0;
        for (int j = 0; j < n; ++j) s = fma(a.A[(size_t)m * a.ld + j], z[j].x, fma(a.B[(size_t)m * a.ld + j], z[j].y, s));
        r[m].x = (T)(E[m] - s);
    }
    __syncthreads();
}

// Points whose fast result is not finite, evaluated densely by the CTA; every
// thread calls it after its outputs are written.  The dense HVP of n >=
// wide_from variables adds its rows in FP64.
template <typename T, typename IO>
__device__ __noinline__ void fp_dense_points(const FpTile<T, IO, true> t, IO *out, int wide_from)
{
    for (int q = 0; q < t.P; ++q) {
        const int n = t.ns[q], z0 = t.base[q];
        IO *o = out + t.xoff[q];
        bool bad = false;
        for (int l = threadIdx.x; l < n; l += kFpThreads) bad |= not_finite((T)o[l]);
        if (!__syncthreads_or(bad)) continue;
        const bool poison = fp_poison<T>(t.a, t.x + t.xoff[q], n);
        fp_residuals<T>(t.a, t.a.E + t.eoff[q], n, t.z + z0, t.rd + z0);
        const FpDense<T> d{t.a.A, t.a.B, t.a.ld, n, t.z + z0, t.rd + z0, poison};
        for (int s = threadIdx.x; s < n; s += kFpThreads)
            o[s] = (IO)dense_row<T>(t.v + t.xoff[q], n, s, n >= wide_from, [&](int i, int j) { return d.entry(i, j); });
        __syncthreads();
    }
}

// ------------------------------------------------------------------ Hessians
// e / n for 0 <= e < 2^32 / n: a multiplication by magic = floor(2^32 / n) + 1
// (n = 1: magic 0).
struct FastDiv {
    unsigned magic;
    __device__ __forceinline__ int div(int e) const { return magic ? (int)__umulhi((unsigned)e, magic) : e; }
};

// The elements of `rows` consecutive Hessian rows of n, out[r n + j] =
// val(r, j), with 16-byte streaming stores where the address allows.  When
// every store lies in one row (n a multiple of the store's values, out aligned)
// vec(r, j, q) gives its values together, with what the row shares read once.
// Every thread of the CTA calls it.
template <typename IO, typename F, typename G>
__device__ __forceinline__ void stream_rows(IO *out, int rows, int n, FastDiv fd, F &&val, G &&vec)
{
    using Vec = typename std::conditional<sizeof(IO) == 8, double2, float4>::type;
    constexpr int V = 16 / (int)sizeof(IO);
    const int cnt = rows * n;
    const int mis = (int)(((16 - ((size_t)out & 15)) & 15) / sizeof(IO));
    const int head = mis < cnt ? mis : cnt, nvec = (cnt - head) / V;
    auto put = [&](int e, const IO(&q)[V]) {
        Vec o;
        if constexpr (V == 2) {
            o.x = q[0];
            o.y = q[1];
        } else {
            o.x = q[0];
            o.y = q[1];
            o.z = q[2];
            o.w = q[3];
        }
        __stcs(reinterpret_cast<Vec *>(out + e), o);
    };
    if (n % V == 0 && head == 0) {
        for (int w = threadIdx.x; w < nvec; w += blockDim.x) {
            const int e = w * V, r = fd.div(e);
            IO q[V];
            vec(r, e - r * n, q);
            put(e, q);
        }
        return;
    }
    auto one = [&](int e) {
        const int r = fd.div(e);
        out[e] = (IO)val(r, e - r * n);
    };
    for (int e = threadIdx.x; e < head; e += blockDim.x) one(e);
    for (int w = threadIdx.x; w < nvec; w += blockDim.x) {
        const int e = head + w * V;
        int r = fd.div(e), j = e - r * n;
        IO q[V];
#pragma unroll
        for (int i = 0; i < V; ++i) {
            q[i] = (IO)val(r, j);
            if (++j == n) {
                j = 0;
                ++r;
            }
        }
        put(e, q);
    }
    for (int e = head + nvec * V + threadIdx.x; e < cnt; e += blockDim.x) one(e);
}

// The Hessian rows [r0, r1) of one point by the dense propagation; the CTA's
// threads take whole rows.
template <typename T, typename IO>
__device__ __noinline__ void ros_dense_rows(const IO *x, IO *H, int n, int r0, int r1)
{
    const RosBad b = ros_bad<T>(x, n);
    for (int i = r0 + (int)threadIdx.x; i < r1; i += blockDim.x)
        for (int j = 0; j < n; ++j) H[(size_t)i * n + j] = (IO)ros_dense_entry<T>(x, n, b, i, j);
}
template <typename T, typename IO>
__device__ __noinline__ void ack_dense_rows(const IO *x, IO *H, int n, int r0, int r1)
{
    const AckDense<T, IO> d(x, n);
    for (int i = r0 + (int)threadIdx.x; i < r1; i += blockDim.x)
        for (int j = 0; j < n; ++j) H[(size_t)i * n + j] = (IO)d.entry(i, j);
}
// z, r: shared scratch of n elements each
template <typename T, typename IO>
__device__ __noinline__ void fp_dense_hessian(const FpArgs a, const IO *x, IO *H, int n, Two<double> *z, Two<T> *r)
{
    __syncthreads();
    const SinCosK k = sincos_k(0);
    for (int l = threadIdx.x; l < n; l += blockDim.x) sincos_rad(k, (double)x[l], z[l].x, z[l].y);
    const bool poison = fp_poison<T>(a, x, n);
    fp_residuals<T>(a, a.E, n, z, r);
    const FpDense<T> d{a.A, a.B, a.ld, n, z, r, poison};
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) H[e] = (IO)d.entry(e / n, e % n);
    __syncthreads();
}

// Fletcher-Powell, f_ij = 2 sum_m J_mi J_mj (+ the curvature on the diagonal):
// a 4 x 4 block of one point's products J^T J in registers, compensated FP32 as
// blocked Sum2 (plain FMAs over kSumBlock rows, then TwoSum), as the dense
// sweep's sum over terms.
template <typename T>
struct Gram4;
template <>
struct Gram4<double> {
    double s[4][4];
    __device__ __forceinline__ void init()
    {
#pragma unroll
        for (int i = 0; i < 16; ++i) s[i / 4][i % 4] = 0.0;
    }
    __device__ __forceinline__ void add(const double *p, const double *q)
    {
        double u[4], w[4];
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
            const double2 a = *reinterpret_cast<const double2 *>(p + i), b = *reinterpret_cast<const double2 *>(q + i);
            u[i] = a.x;
            u[i + 1] = a.y;
            w[i] = b.x;
            w[i + 1] = b.y;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) s[i][j] = __fma_rn(u[i], w[j], s[i][j]);
    }
    __device__ __forceinline__ void flush() {}
    __device__ __forceinline__ double value(int i, int j) const { return 2.0 * s[i][j]; }
};
template <>
struct Gram4<float> {
    CSum s[4][4];
    float p[4][4];
    __device__ __forceinline__ void init()
    {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            s[i / 4][i % 4] = CSum{0.f, 0.f};
            p[i / 4][i % 4] = 0.f;
        }
    }
    __device__ __forceinline__ void add(const float *a, const float *b)
    {
        const float4 x = *reinterpret_cast<const float4 *>(a), y = *reinterpret_cast<const float4 *>(b);
        const float u[4] = {x.x, x.y, x.z, x.w};
        const float w[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) vfma(u[i], w, p[i]);
    }
    // csum_add of two neighbours at a time (packed; a - b as the exact
    // fma(-1, b, a), each component rounding as csum_add's)
    __device__ __forceinline__ void flush()
    {
        const float2 m1 = make_float2(-1.f, -1.f);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; j += 2) {
                const float2 a = make_float2(s[i][j].s, s[i][j + 1].s), b = make_float2(p[i][j], p[i][j + 1]);
                const float2 e = make_float2(s[i][j].e, s[i][j + 1].e);
                const float2 t = __fadd2_rn(a, b), bb = __ffma2_rn(m1, a, t);
                const float2 x = __ffma2_rn(m1, __ffma2_rn(m1, bb, t), a), y = __ffma2_rn(m1, bb, b);
                const float2 f = __fadd2_rn(e, __fadd2_rn(x, y));
                s[i][j] = CSum{t.x, f.x};
                s[i][j + 1] = CSum{t.y, f.y};
                p[i][j] = p[i][j + 1] = 0.f;
            }
    }
    __device__ __forceinline__ float value(int i, int j) const { return 2.0f * csum_value(s[i][j]); }
};

// J_mj = A_mj cos x_j - B_mj sin x_j, as the dense sweep rounds it
template <typename T>
__device__ __forceinline__ T fp_jacobian(T a, T b, T s, T c)
{
    return fma_(b, -s, a * c);
}

}  // namespace chessfad
