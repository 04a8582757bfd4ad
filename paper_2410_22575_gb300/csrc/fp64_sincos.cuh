// fp64_sincos.cuh -- sin and cos of one FP64 argument with about 20 FP64
// instructions and register operands.
//
// The FP64 pipe issues one warp instruction per 16 clocks and SM, so the
// structured kernels are bound by their FP64 instruction counts, of which sin
// and cos of the variables are the largest part.  A DFMA with a literal
// operand issues at 84 % of the pipe's rate (chessfad_peak_operand_rates), so
// the coefficients are read from device memory into registers once per thread.
//
// sin t = t + t z P(z), cos t = 1 + z Q(z), z = t^2, |t| <= pi/4, with P of
// degree 5 and Q of degree 6: the minimax polynomials of the relative error by
// the Remez exchange (60-digit arithmetic), 3.6e-18 and 3.9e-20.  The argument
// is reduced to |t| <= pi/4 by subtracting the nearest multiple of pi/2,
// rounded to an integer by adding and subtracting 1.5 * 2^52, with pi/2 as the
// sum of three doubles (Cody and Waite) or, for sin and cos of 2 pi x, exactly.
// Arguments beyond the reduction's range, Inf and NaN go to the CUDA functions
// (the test is on the exponent bits: an FP64 comparison is an FP64 instruction).
#pragma once

#include <cuda_runtime.h>

namespace chessfad {

struct SinCosK {
    double p[6], q[7];  // P, Q
    double lo;          // sin of 2 pi x: 2 pi minus its double
};

// {radians, turns}; the turn coefficients are the radian ones times (2 pi)^k
static __device__ __align__(16) double g_sincos_k[2][14] = {
    {-0.1666666666666663072846, 0.008333333333322118472083, -0.000198412698295895012389, 0.000002755731362138341424732,
     -2.505074776343208191249e-8, 1.589623022002321512473e-10, -0.4999999999999999950985, 0.04166666666666646985499,
     -0.001388888888886200048839, 0.00002480158728409487675042, -2.755731311735106821715e-7, 2.087558213418349774362e-9,
     -1.135328159075634913976e-11, 0.0},
    {-41.34170224039967108917, 81.60524927596523121765, -76.70585970790547941786, 42.05868539406072540225,
     -15.09382276147644805653, 3.781224233231761639491, -19.73920880217871704417, 64.93939402266798475102,
     -85.45681720652828634291, 60.24464132938644196631, -26.42625092738025708265, 7.903091594438964991843,
     -1.696834816336523887832, 2.449293598294706354452e-16}};

__device__ __forceinline__ SinCosK sincos_k(int turns)
{
    SinCosK k;
    const double *g = g_sincos_k[turns];
    auto at = [&](int i, double &a, double &b) {
        asm("{\n\t.reg .u64 ga;\n\tcvta.to.global.u64 ga, %2;\n\tld.global.nc.v2.f64 {%0, %1}, [ga];\n\t}"
            : "=d"(a), "=d"(b)
            : "l"(g + i));
    };
    at(0, k.p[0], k.p[1]);
    at(2, k.p[2], k.p[3]);
    at(4, k.p[4], k.p[5]);
    at(6, k.q[0], k.q[1]);
    at(8, k.q[2], k.q[3]);
    at(10, k.q[4], k.q[5]);
    at(12, k.q[6], k.lo);
    return k;
}

// s, c of quadrant number k from sin and cos of the reduced argument
__device__ __forceinline__ void sincos_quadrant(int k, double sr, double cr, double &s, double &c)
{
    const double a = k & 1 ? cr : sr, b = k & 1 ? sr : cr;
    s = __hiloint2double(__double2hiint(a) ^ ((k & 2) << 30), __double2loint(a));
    c = __hiloint2double(__double2hiint(b) ^ (((k + 1) & 2) << 30), __double2loint(b));
}

__device__ __forceinline__ double sincos_q(const SinCosK &k, double z)
{
    double q = k.q[6];
#pragma unroll
    for (int i = 5; i >= 0; --i) q = __fma_rn(q, z, k.q[i]);
    return __fma_rn(q, z, 1.0);
}
__device__ __forceinline__ double sincos_p(const SinCosK &k, double z)
{
    double p = k.p[5];
#pragma unroll
    for (int i = 4; i >= 0; --i) p = __fma_rn(p, z, k.p[i]);
    return p;
}

constexpr double kRoundMagic = 6755399441055744.0;  // 1.5 * 2^52

// sin x, cos x
__device__ __forceinline__ void sincos_rad(const SinCosK &k, double x, double &s, double &c)
{
    if (((unsigned)__double2hiint(x) & 0x7fffffffu) >= 0x40f00000u) {  // |x| >= 65536, Inf, NaN
        sincos(x, &s, &c);
        return;
    }
    const double m = __fma_rn(x, 0.63661977236758134308, kRoundMagic), t = m - kRoundMagic;
    double r = __fma_rn(t, -1.570796326794896557999, x);
    r = __fma_rn(t, -6.123233995736766035869e-17, r);
    r = __fma_rn(t, 1.497384904859169832944e-33, r);
    const double z = r * r;
    sincos_quadrant(__double2loint(m), __fma_rn(r * z, sincos_p(k, z), r), sincos_q(k, z), s, c);
}

// sin 2 pi x, cos 2 pi x.  4x + 1.5 * 2^52 rounds to an integer while it lies
// between 2^52 and 2^53, that is for |4x| <= 2^51.
__device__ __forceinline__ void sincos_turn(const SinCosK &k, double x, double &s, double &c)
{
    if (((unsigned)__double2hiint(x) & 0x7fffffffu) >= 0x43000000u) {  // |x| >= 2^49, Inf, NaN
        sincospi(2.0 * x, &s, &c);
        return;
    }
    const double m = __fma_rn(x, 4.0, kRoundMagic), t = m - kRoundMagic;
    const double r = __fma_rn(t, -0.25, x), z = r * r;
    const double q = __fma_rn(sincos_p(k, z), z, k.lo);
    sincos_quadrant(__double2loint(m), __fma_rn(r, 6.283185307179586, r * q), sincos_q(k, z), s, c);
}

}  // namespace chessfad
