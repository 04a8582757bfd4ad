// user_kernel.cuh -- CHESS-VEC (Alg. 7) and CHUNK-HESS (Alg. 5) over a batch
// of points for a user-supplied function.  Compiled at run time (NVRTC) after
// the user's source, with
//   CHESSFAD_USER_T    float or double (the arithmetic precision)
//   CHESSFAD_USER_C    the chunk size (compile-time: the hDual lives in registers)
//   CHESSFAD_USER_FN   the name of the user's function template
//                        template <class R, class X>
//                        R name(const X &x, int n, const double *params);
//   CHESSFAD_USER_DIR  1: the directional kernel only, 0: the others
// Two decompositions:
//  plain (CHESS-VEC / CHUNK-HESS, the paper's L2 over rows, Sec. VI): one
//    thread per (point, row i), sweeping the row's ceil(n/C) chunks; a CTA
//    stages the x (and v) of the points its rows belong to in shared memory;
//  symmetric (SC-HESS-VEC, Alg. 8 / SCHUNK-HESS, Alg. 6): a CTA holds maxpts
//    points with tpp threads each; a point's items (row i, chunk cn >=
//    floor(i/C)) are dealt round-robin to its threads.  The Hessian writes
//    each chunk and its mirror image; the HVP stages the chunks in shared
//    memory (compact upper-block layout) and, after one barrier, every thread
//    sums whole rows, each off-diagonal-chunk entry serving both r_i and r_j;
//  directional (HVP, the default): one thread per (point, chunk), a single
//    evaluation with d1 seeded by v gives the chunk's rows of H v (ceil(n/C)
//    evaluations per point instead of n ceil(n/C)), on numbers that skip the
//    zero components of what does not depend on the chunk; rows that are not
//    finite, and points whose d1 or v is not, are evaluated again by the plain
//    method.
// FP32: the row-times-v products are summed as a Dot2 (TwoProd by FMA plus
// TwoSum), the directional d1 and h carry their errors the same way (Dir); the
// rest of the function's own arithmetic is plain FP32, as written by the
// user, except at n = 1 (FP64 arithmetic, float I/O).  FP64: fused
// multiply-add accumulation.
#pragma once

#include "sym_layout.cuh"
#include "user_num.cuh"

namespace chessfad {
namespace user {

struct UserArgs {
    const void *x;
    const void *v;
    void *out;
    long long batch;
    const double *params;
    int n;
    int maxpts;  // plain: points staged per CTA, min(batch, (blockDim - 1) / n + 2);
                 // symmetric: points per CTA
    int tpp;     // symmetric: threads per point
    int acc;     // symmetric HVP: 0 = stage the chunk matrix, 1 = FP64 row accumulators
};

template <typename T>
struct RowDot;
template <>
struct RowDot<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double a, double b) { s = __fma_rn(a, b, s); }
    __device__ __forceinline__ double value() const { return s; }
};
template <>
struct RowDot<float> {
    CSum s{0.f, 0.f};
    __device__ __forceinline__ void add(float a, float b) { cdot_add(s, a, b); }
    __device__ __forceinline__ float value() const { return csum_value(s); }
};

// T: the arithmetic type; IO: the element type of x, v and the output (IO =
// T except for the one-variable kernels of an FP32 handle, which compute in
// FP64 with float inputs and outputs).
template <typename T, typename IO, int C, bool HVP>
__device__ __forceinline__ void user_sweep(const UserArgs &a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *xs = reinterpret_cast<T *>(smem_raw);
    T *vs = xs + (size_t)a.maxpts * a.n;
    const int n = a.n;
    const long long items = a.batch * n;
    const long long first = (long long)blockIdx.x * blockDim.x;
    const long long last = (first + blockDim.x <= items ? first + blockDim.x : items) - 1;
    const long long p0 = first / n;
    const int staged = (int)(last / n - p0 + 1) * n;
    const IO *xg = static_cast<const IO *>(a.x) + p0 * n;
    const IO *vg = static_cast<const IO *>(a.v) + p0 * n;
    for (int t = threadIdx.x; t < staged; t += blockDim.x) {
        xs[t] = (T)xg[t];
        if (HVP) vs[t] = (T)vg[t];
    }
    __syncthreads();
    const long long item = first + threadIdx.x;
    if (item >= items) return;
    const long long p = item / n;
    const int i = (int)(item - p * n);
    const T *xp = xs + (p - p0) * n;
    const T *vp = vs + (p - p0) * n;
    const SeedK<T> z = seed_constants<T>();
    const int nch = (n + C - 1) / C;
    RowDot<T> dot;
    for (int cn = 0; cn < nch; ++cn) {
        const int cstart = cn * C;
        const Vars<T, C> x{xp, i, cstart, z};
        const Num<T, C> r = ::CHESSFAD_USER_FN<Num<T, C>, Vars<T, C>>(x, n, a.params);
        if (HVP) {
#pragma unroll
            for (int l = 0; l < C; ++l)
                if (cstart + l < n) dot.add(r.a.h[l], vp[cstart + l]);
        } else {
            IO *H = static_cast<IO *>(a.out) + (p * n + i) * (long long)n + cstart;
#pragma unroll
            for (int l = 0; l < C; ++l)
                if (cstart + l < n) H[l] = (IO)r.a.h[l];
        }
    }
    if (HVP) static_cast<IO *>(a.out)[p * n + i] = (IO)dot.value();
}

template <typename T, int C, bool HVP>
__device__ __forceinline__ void user_sym(const UserArgs &a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n, ppb = a.maxpts, tpp = a.tpp;
    // accumulators first (8-byte aligned), then x, v and the staged chunks
    // (accumulator form: the per-iteration stage, SymStage, in their place)
    double *accs = reinterpret_cast<double *>(smem_raw);
    const bool acc_form = HVP && a.acc;
    T *xs = reinterpret_cast<T *>(smem_raw + (acc_form ? (size_t)ppb * n * sizeof(double) : 0));
    T *vs = xs + (size_t)ppb * n;
    T *hs = vs + (HVP ? (size_t)ppb * n : 0);
    const long long p0 = (long long)blockIdx.x * ppb;
    const int npts = (int)(a.batch - p0 < ppb ? a.batch - p0 : ppb);
    const T *xg = static_cast<const T *>(a.x) + p0 * n;
    const T *vg = static_cast<const T *>(a.v) + p0 * n;
    for (int e = threadIdx.x; e < npts * n; e += blockDim.x) {
        xs[e] = xg[e];
        if (HVP) vs[e] = vg[e];
        if (acc_form) accs[e] = 0.0;
    }
    __syncthreads();
    const int q = threadIdx.x / tpp, t = threadIdx.x - q * tpp;
    double *acc = accs + (size_t)q * n;
    const bool active = q < npts;
    const long long p = p0 + q;
    const T *xp = xs + (size_t)q * n;
    T *Hs = hs + (size_t)q * sym_hs_elems(n, C);
    const SeedK<T> z = seed_constants<T>();
    const int nch = (n + C - 1) / C;
    const int items = C * nch * (nch + 1) / 2;
    if (HVP && acc_form) {
        // Alg. 8's two updates (r_i += sum_l H_il v_l; off the diagonal chunk
        // also r_l += H_il v_i) in FP64, reproducibly: each iteration stages
        // every thread's chunk and row dot (SymStage), and each thread adds
        // the contributions to its own rows in thread order.  Every thread
        // runs the same number of iterations (the barriers).
        const size_t soff = ((size_t)(reinterpret_cast<unsigned char *>(hs) - smem_raw) + 15) / 16 * 16;
        const SymStage<T, C> stage(smem_raw + soff, (int)blockDim.x);
        const T *vp = vs + (size_t)q * n;
        const int iters = (items + tpp - 1) / tpp;
        for (int it = 0; it < iters; ++it) {
            const int k = t + it * tpp;
            int i = -1, cn = 0;
            T h[C];
            double own = 0.0;
            if (active && k < items) {
                sym_item(k, C, nch, i, cn);
                if (i >= n) i = -1;
            }
            if (i >= 0) {
                const int cstart = cn * C;
                const Vars<T, C> x{xp, i, cstart, z};
                const Num<T, C> r = ::CHESSFAD_USER_FN<Num<T, C>, Vars<T, C>>(x, n, a.params);
#pragma unroll
                for (int l = 0; l < C; ++l) {
                    h[l] = r.a.h[l];
                    if (cstart + l < n) own = fma((double)h[l], (double)vp[cstart + l], own);
                }
            } else {
#pragma unroll
                for (int l = 0; l < C; ++l) h[l] = T(0);
            }
            stage.put(threadIdx.x, h, own, i, cn);
            __syncthreads();
            if (active) {
                const int t0 = q * tpp;
                for (int srow = t; srow < n; srow += tpp) {
                    const int scn = srow / C, sl = srow - scn * C;
                    double sum = acc[srow];
                    for (int u = 0; u < tpp; ++u) {
                        const int ui = stage.row(t0 + u);
                        if (ui < 0) continue;
                        if (ui == srow) sum += stage.own(t0 + u);
                        const int ucn = stage.chunk(t0 + u);
                        if (ucn == scn && ucn > ui / C) sum += (double)stage.h(t0 + u, sl) * (double)vp[ui];
                    }
                    acc[srow] = sum;
                }
            }
            __syncthreads();
        }
    }
    for (int k = (active && !(HVP && acc_form)) ? t : items; k < items; k += tpp) {
        int i = 0, cn = 0;
        sym_item(k, C, nch, i, cn);
        if (i >= n) continue;
        const int cstart = cn * C;
        const Vars<T, C> x{xp, i, cstart, z};
        const Num<T, C> r = ::CHESSFAD_USER_FN<Num<T, C>, Vars<T, C>>(x, n, a.params);
        if (HVP) {
            T *hrow = Hs + sym_hs_row(i, n, C) - (i / C) * C;
#pragma unroll
            for (int l = 0; l < C; ++l)
                if (cstart + l < n) hrow[cstart + l] = r.a.h[l];
        } else {
            T *H = static_cast<T *>(a.out) + (size_t)p * n * n;
            const bool mirror = cn > i / C;
#pragma unroll
            for (int l = 0; l < C; ++l) {
                const int j = cstart + l;
                if (j < n) {
                    H[(size_t)i * n + j] = r.a.h[l];
                    if (mirror) H[(size_t)j * n + i] = r.a.h[l];
                }
            }
        }
    }
    if (HVP) {
        // r_s = sum_j H_sj v_j: entries right of row s's diagonal chunk from
        // row s, entries left of it from column s (H_sj = H_js).
        __syncthreads();
        if (active && acc_form) {
            T *O = static_cast<T *>(a.out) + p * n;
            for (int srow = t; srow < n; srow += tpp) O[srow] = (T)acc[srow];
        } else if (active) {
            const T *vp = vs + (size_t)q * n;
            T *O = static_cast<T *>(a.out) + p * n;
            for (int srow = t; srow < n; srow += tpp) {
                const int dstart = (srow / C) * C;
                const T *own = Hs + sym_hs_row(srow, n, C) - dstart;
                RowDot<T> dot;
                for (int j = 0; j < dstart; ++j) dot.add(Hs[sym_hs_row(j, n, C) + srow - (j / C) * C], vp[j]);
                for (int j = dstart; j < n; ++j) dot.add(own[j], vp[j]);
                O[srow] = dot.value();
            }
        }
    }
}

// Rows cstart .. cstart + C - 1 of H v by the plain method (Alg. 7).
template <typename T, int C>
__device__ __noinline__ void user_dense_rows(const T *xp, const T *vp, T *out, int n, int cstart, const double *params)
{
    const SeedK<T> z = seed_constants<T>();
    for (int i = cstart; i < cstart + C && i < n; ++i) {
        RowDot<T> dot;
        for (int c0 = 0; c0 < n; c0 += C) {
            const Vars<T, C> x{xp, i, c0, z};
            const Num<T, C> r = ::CHESSFAD_USER_FN<Num<T, C>, Vars<T, C>>(x, n, params);
#pragma unroll
            for (int l = 0; l < C; ++l)
                if (c0 + l < n) dot.add(r.a.h[l], vp[c0 + l]);
        }
        out[i] = dot.value();
    }
}

// A CTA holds a.maxpts points (a power of two <= 32, one per lane) and
// blockDim / maxpts of their chunks; x and v of its points are staged in
// shared memory point by point within each variable, so a warp's lanes read
// different banks.  Lanes of a warp are on the same chunk (or on a few), so
// the activity of their numbers agrees and its branches do not diverge.
// Bound by the arithmetic of f: its functions of values, once per chunk, and the
// active components.  The extended-operator test function, n = 64, C = 8, FP64,
// 4096 points: symmetric method 100.7 ms; every component of every number 2.83
// ms; active components 1.67 ms; two powers instead of three in an inactive
// pow() 1.30 ms.
// FP32: 81 us with plain sums over v (C = 8), whose rms error was up to 1.27 times
// the symmetric method's and grew with n; with Dir's (0.6 to 1.0 times) 143 us one
// component at a time, 130 two at a time (C = 4; the symmetric method takes 1555).
template <typename T, int C>
__device__ __forceinline__ void user_directional(const UserArgs &a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n, nch = (n + C - 1) / C, L = a.maxpts, slots = blockDim.x / L;
    const int groups = (nch + slots - 1) / slots;
    const long long p0 = (long long)(blockIdx.x / groups) * L;
    const int npts = (int)(a.batch - p0 < L ? a.batch - p0 : L);
    const int S = L + 1;  // odd: the transposing stores hit different banks
    T *xs = reinterpret_cast<T *>(smem_raw), *vs = xs + (size_t)n * S;
    const T *xg = static_cast<const T *>(a.x) + p0 * n, *vg = static_cast<const T *>(a.v) + p0 * n;
    for (int e = threadIdx.x; e < npts * n; e += blockDim.x) {
        const int q = e / n, k = e - q * n;
        xs[k * S + q] = xg[e];
        vs[k * S + q] = vg[e];
    }
    __syncthreads();
    const int q = threadIdx.x & (L - 1);
    const int cn = (int)(blockIdx.x % groups) * slots + threadIdx.x / L, cstart = cn * C;
    if (q >= npts || cn >= nch) return;
    using N = Num<T, C, true>;
    const DirVars<T, C> x{xs + q, vs + q, S, cstart, seed_constants<T>()};
    const N r = ::CHESSFAD_USER_FN<N, DirVars<T, C>>(x, n, a.params);
    T *out = static_cast<T *>(a.out) + (p0 + q) * n;
    // stays 0 while the chunk's rows, d1 (which every skipped product's
    // factors reach) and v are finite
    T zero = r.a.d1.value() * T(0);
#pragma unroll
    for (int l = 0; l < C; ++l) {
        if (cstart + l < n) {
            const T h = r.act ? r.a.h[l].value() : T(0);
            out[cstart + l] = h;
            zero += h * T(0);
        }
    }
    for (int k = 0; k < n; ++k) zero += vs[k * S + q] * T(0);
    if (!(zero == T(0)))
        user_dense_rows<T, C>(xg + (size_t)q * n, vg + (size_t)q * n, out, n, cstart, a.params);
}

}  // namespace user
}  // namespace chessfad

// CHESSFAD_USER_DIR: the directional kernel, else the row methods; the two are
// compiled as two programs at the same time.
#if CHESSFAD_USER_DIR

extern "C" __global__ void __launch_bounds__(256) chessfad_user_dir_hvp(chessfad::user::UserArgs a)
{
    chessfad::user::user_directional<CHESSFAD_USER_T, CHESSFAD_USER_C>(a);
}

#else

extern "C" __global__ void __launch_bounds__(256) chessfad_user_sym_hvp(chessfad::user::UserArgs a)
{
    chessfad::user::user_sym<CHESSFAD_USER_T, CHESSFAD_USER_C, true>(a);
}

extern "C" __global__ void __launch_bounds__(256) chessfad_user_sym_hessian(chessfad::user::UserArgs a)
{
    chessfad::user::user_sym<CHESSFAD_USER_T, CHESSFAD_USER_C, false>(a);
}

extern "C" __global__ void __launch_bounds__(256) chessfad_user_hvp(chessfad::user::UserArgs a)
{
    chessfad::user::user_sweep<CHESSFAD_USER_T, CHESSFAD_USER_T, CHESSFAD_USER_C, true>(a);
}

extern "C" __global__ void __launch_bounds__(256) chessfad_user_hessian(chessfad::user::UserArgs a)
{
    chessfad::user::user_sweep<CHESSFAD_USER_T, CHESSFAD_USER_T, CHESSFAD_USER_C, false>(a);
}

#if CHESSFAD_USER_F32
// One variable in an FP32 handle: the Hessian is a single entry, a sum of
// terms that can cancel far below their size, so no FP32 evaluation bounds
// its relative error; it is computed in FP64 with float x, v and output.
extern "C" __global__ void __launch_bounds__(256) chessfad_user_hvp_n1(chessfad::user::UserArgs a)
{
    chessfad::user::user_sweep<double, float, 1, true>(a);
}

extern "C" __global__ void __launch_bounds__(256) chessfad_user_hessian_n1(chessfad::user::UserArgs a)
{
    chessfad::user::user_sweep<double, float, 1, false>(a);
}
#endif

#endif
