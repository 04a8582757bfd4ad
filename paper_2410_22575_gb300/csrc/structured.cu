// structured.cu -- kernels and launches of the structured evaluation over a
// contiguous batch (structured.cuh).
//
// H v through the default call, GB300, dense symmetric method -> here:
//   Ackley n = 64, FP64, 65536 points            102.2 ms -> 0.256 ms
//   Ackley n = 64, FP32-comp, 524288 points       15.9 ms -> 0.119 ms
//   Fletcher-Powell n = 32, FP32-comp, 16384       1.83 ms -> 0.086 ms
//   Fletcher-Powell n = 75, FP64, 1000            151.7 ms -> 0.115 ms
// Hessians:
//   Rosenbrock n = 256, FP64, 1024                 86.1 ms -> 0.076 ms (7.0 TB/s written)
//   Ackley n = 33, FP32-comp, 20000                0.178 ms -> 0.035 ms
//   Fletcher-Powell n = 48, FP32-comp, 4096        2.23 ms -> 0.107 ms
// The Rosenbrock kernels stream.  In FP64 the others are bound by the FP64 pipe
// (sin, cos and the sums under sqrt and exp; the residuals), and so are the
// Fletcher-Powell ones in compensated FP32; Ackley's H v there is bound by
// instruction issue and its Hessian by shared-memory loads.  The FP64 pipe takes
// one warp instruction per 16 clocks and SM, so what is not FP64 arithmetic stays
// off it: conversions and tests of FP64 values run on 32-bit words, coefficients
// come from registers (fp64_sincos.cuh).
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "structured.cuh"
#include "structured.h"
#include "structured_tune.h"

namespace chessfad {
namespace {

constexpr int kThreads = 256;
constexpr int kAckThreads = 128;  // small CTAs: the last round of CTAs is short
constexpr long long kMaxBlocks = 0x7fffffffLL;

// A group of G lanes per point.  FP32: x and v streamed once, neighbours from
// L1; FP64: 11 FP64 instructions per variable are the bound from a few hundred
// thousand variables on (n = 256, 1024 points: 13.6 us, FP64 pipe 58 % busy,
// the launch and its tail the rest).
template <typename T, typename IO>
__global__ void __launch_bounds__(kThreads) ros_hvp_kernel(const StructArgs a, int G)
{
    const long long p = ((long long)blockIdx.x * kThreads + threadIdx.x) / G;
    const int t = threadIdx.x & (G - 1);
    const bool active = p < a.batch;
    const size_t o = active ? (size_t)p * a.n : 0;
    ros_point<T, IO>(static_cast<const IO *>(a.x) + o, static_cast<const IO *>(a.v) + o, static_cast<IO *>(a.out) + o,
                     a.n, t, G, active, a.wide);
}

// A group of G lanes per point, EPL variables per lane in registers, no shared
// memory and no barrier.  n = 64: FP64, 65536 points, 258 us with the FP64 pipe
// 85 % busy (3512 operations a point, 183 us of it at its peak); FP32-comp,
// 524288 points, 119 us, instruction issue 75 % busy (59 us of HBM traffic).
template <typename T, typename IO, int EPL, bool kVec = false>
__global__ void __launch_bounds__(kAckThreads) ack_hvp_kernel(const StructArgs a, int G, const AckConst nc)
{
    const long long p = ((long long)blockIdx.x * kAckThreads + threadIdx.x) / G;
    const int t = threadIdx.x & (G - 1);
    const bool active = p < a.batch;
    const size_t o = active ? (size_t)p * a.n : 0;
    ack_point<T, IO, EPL, kVec>(static_cast<const IO *>(a.x) + o, static_cast<const IO *>(a.v) + o,
                          static_cast<IO *>(a.out) + o, a.n, t, G, active, a.wide, nc);
}

// One FpTile per CTA.  FP64 pipe: n = 32, 16384 points, FP64 254 us (97 % busy),
// FP32-comp 86 us (89 %: two FMAs per (m, j) for the residual, 20 instructions
// per variable for sin and cos); n = 75, 1000 points, FP64 115 us (250 CTAs on
// 152 SMs).
template <typename T, typename IO, bool kWide>
__global__ void __launch_bounds__(kFpThreads) fp_hvp_kernel(const StructArgs a, const FpShape sh, int ppb)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n;
    const long long p0 = (long long)blockIdx.x * ppb;
    const int P = (int)min((long long)ppb, a.batch - p0);
    const FpArgs fa{a.A, a.B, a.E, a.ld};
    IO *out = static_cast<IO *>(a.out);
    FpTile<T, IO, true> tile(fa, static_cast<const IO *>(a.x), static_cast<const IO *>(a.v), smem_raw, sh, P, P * n);
    for (int q = threadIdx.x; q <= P; q += kFpThreads) {
        tile.base[q] = q * n;
        if (q < P) {
            tile.ns[q] = n;
            tile.xoff[q] = (p0 + q) * n;
            tile.eoff[q] = 0;
        }
    }
    __syncthreads();
    FpSums<T, 2> sums[kFpNpt];
    tile.template run<kWide>(0, n, sums);
    bool bad = false;
#pragma unroll
    for (int i = 0; i < kFpNpt; ++i) {
        const int u = threadIdx.x + i * kFpThreads;
        if (u >= P * n) break;
        const FpSums<T, 2> &f = sums[i];
        const T o = tile.combine(u, f.value(0), f.value(1), f.value(2), f.value(3));
        bad |= not_finite(o);
        out[p0 * n + u] = (IO)o;
    }
    if (__syncthreads_or(bad)) fp_dense_points<T, IO>(tile, out, a.wide ? 0 : n + 1);
}

// ---- Hessians

// `rows` rows of the batch's row space per CTA; a row has three entries, the
// rest of it is the zeros of the terms' independent variables.  Bound by the
// stores: n = 256, 1024 points, FP64 76 us (7.0 TB/s), FP32-comp 39 us.
template <typename T, typename IO>
__global__ void __launch_bounds__(kThreads) ros_hessian_kernel(const StructArgs a, int rows, FastDiv fd)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n;
    const long long row0 = (long long)blockIdx.x * rows, total = a.batch * n;
    const int cnt = (int)min((long long)rows, total - row0);
    T *lo = reinterpret_cast<T *>(smem_raw), *diag = lo + rows, *up = diag + rows;
    short *ls = reinterpret_cast<short *>(up + rows);
    const long long p0 = row0 / n;
    const int l0 = (int)(row0 - p0 * n);
    const int npts = (l0 + cnt - 1) / n + 1;
    const IO *x = static_cast<const IO *>(a.x) + p0 * n;  // the first touched point
    IO *H = static_cast<IO *>(a.out) + (size_t)row0 * n;
    bool bad = false;
    for (int e = threadIdx.x; e < npts * n; e += kThreads) {
        const int l = e - fd.div(e) * n, r = e - l0;
        const T x0 = (T)x[e], xp = l + 1 < n ? (T)x[e + 1] : T(0);
        if (l + 1 < n) bad |= not_finite(x0) || not_finite(T(200) * fma_(T(-1), x0 * x0, xp));
        if (r >= 0 && r < cnt) {
            const RosRow<T> w = ros_row<T>(l > 0 ? (T)x[e - 1] : T(0), x0, xp, l, n);
            lo[r] = w.lo;
            diag[r] = w.diag;
            up[r] = w.up;
            ls[r] = (short)l;
            bad |= not_finite(w.diag) || not_finite(w.up);
        }
    }
    if (__syncthreads_or(bad)) {  // dense propagation (equal to the rows below for finite points)
        for (int q = 0; q < npts; ++q) {
            const int r0 = max(0, l0 - q * n), r1 = min(n, l0 + cnt - q * n);
            ros_dense_rows<T, IO>(x + (size_t)q * n, static_cast<IO *>(a.out) + (size_t)(p0 + q) * n * n, n, r0, r1);
        }
        return;
    }
    auto val = [&](int r, int j) {
        const int d = j - ls[r] + 1;
        T v = T(0);
        if ((unsigned)d <= 2u) v = d == 1 ? diag[r] : d == 2 ? up[r] : lo[r];
        return v;
    };
    stream_rows(H, cnt, n, fd, val, [&](int r, int j, IO *q) {
        const int d = j - ls[r];  // -1, 0, 1: the row's entries
        const T a0 = lo[r], a1 = diag[r], a2 = up[r];
#pragma unroll
        for (int i = 0; i < 16 / (int)sizeof(IO); ++i)
            q[i] = (IO)(d + i == -1 ? a0 : d + i == 0 ? a1 : d + i == 1 ? a2 : T(0));
    });
}

// ppc whole points per CTA, or, split > 1, one of `split` parts of one
// point's rows.  Entry (i, j) is (K x_i) x_j + (G s_i) s_j, K = p1 r2 + p2 r1^2
// and G = q2 the second derivatives of the tail in its two sums, s = sin 2 pi x;
// the diagonal adds p1 r1 + q1 cos 2 pi x.  Bound by the shared-memory loads
// per element (n = 33, FP32-comp: 76 % busy, issue 60 %, 2.5 TB/s written).
template <typename T, typename IO>
__global__ void __launch_bounds__(kThreads) ack_hessian_kernel(const StructArgs a, int ppc, int split, FastDiv fd,
                                                               const AckConst nc)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    struct alignas(2 * sizeof(T)) Pair {
        T x, s;
    };
    const int n = a.n;
    const long long p0 = split > 1 ? blockIdx.x / split : (long long)blockIdx.x * ppc;
    const int part = split > 1 ? (int)(blockIdx.x % split) : 0;
    const int npts = (int)min((long long)ppc, a.batch - p0), nv = npts * n;
    const int r0 = n * part / split, r1 = split > 1 ? n * (part + 1) / split : nv;
    Pair *xs = reinterpret_cast<Pair *>(smem_raw);  // x_j, s_j of every variable
    Pair *ab = xs + ppc * n;                        // K x_i, G s_i
    T *dg = reinterpret_cast<T *>(ab + ppc * n);    // cos 2 pi x_i, then the diagonal's addition
    double *sums = reinterpret_cast<double *>(smem_raw + align_up((size_t)ppc * n * 5 * sizeof(T), 16));
    int *flag = reinterpret_cast<int *>(sums + 2 * ppc);
    const IO *x = static_cast<const IO *>(a.x) + p0 * n;
    const int tid = threadIdx.x;
    const Turn<T> turn;
    for (int u = tid; u < nv; u += kThreads) {
        T s, c;
        const T xv = (T)x[u];
        turn(xv, s, c);
        xs[u].x = xv;
        xs[u].s = s;
        dg[u] = c;
    }
    for (int q = tid; q < npts; q += kThreads) flag[q] = 0;
    __syncthreads();
    // S and C of each point in FP64, G lanes per point: few, so that few FP64
    // additions go across lanes, but at most 16 variables per lane
    const int G = n <= 8 ? 1 : n <= 128 ? 8 : 32, lane = tid & (G - 1);
    for (int b = 0; b < npts; b += kThreads / G) {
        const int q = b + tid / G;
        double S = 0.0, C = 0.0;
        for (int k = lane; k < n && q < npts; k += G) {
            const double xd = widen(xs[q * n + k].x);
            S = fma(xd, xd, S);
            C += widen(dg[q * n + k]);
        }
        for (int off = G >> 1; off > 0; off >>= 1) {
            S += __shfl_xor_sync(0xffffffffu, S, off);
            C += __shfl_xor_sync(0xffffffffu, C, off);
        }
        if (q < npts && lane == 0) {
            sums[2 * q] = S;
            sums[2 * q + 1] = C;
        }
    }
    __syncthreads();
    // the tail's factors, one thread per point
    T *tail = reinterpret_cast<T *>(flag + ppc + (ppc & 1));
    for (int q = tid; q < npts; q += kThreads) {
        const AckTail<T> k = ack_tail(sums[2 * q], sums[2 * q + 1], nc, false, T(0));
        const double p1 = k.p1, r1 = k.r1;  // FP64: the factors are shared by every entry
        tail[4 * q] = (T)fma(p1, (double)k.r2, ((double)k.p2 * r1) * r1);
        tail[4 * q + 1] = k.q2;
        tail[4 * q + 2] = (T)(p1 * r1);
        tail[4 * q + 3] = k.q1;
    }
    __syncthreads();
    for (int u = tid; u < nv; u += kThreads) {
        const int q = fd.div(u);
        const Pair e = xs[u];
        Pair f;
        f.x = tail[4 * q] * e.x;
        f.s = tail[4 * q + 1] * e.s;
        const T d = fma_(tail[4 * q + 3], dg[u], tail[4 * q + 2]);
        ab[u] = f;
        dg[u] = d;
        if (not_finite(e.x) || not_finite(f.x) || not_finite(f.s) || not_finite(d)) atomicOr(&flag[q], 1);
    }
    __syncthreads();
    IO *H = static_cast<IO *>(a.out) + ((size_t)p0 * n + r0) * n;
    // The smaller index's factors are the scaled ones, so H is symmetric bit
    // for bit.
    auto val = [&](int r, int j) {
        const int u = r + r0, w = (split > 1 ? 0 : fd.div(u) * n) + j;
        const Pair e = (w < u ? ab : xs)[w], f = (w < u ? xs : ab)[u];
        T v = fma_(f.x, e.x, f.s * e.s);
        if (w == u) v += dg[u];
        return v;
    };
    stream_rows(H, r1 - r0, n, fd, val, [&](int r, int j, IO *q) {
        const int u = r + r0, w = (split > 1 ? 0 : fd.div(u) * n) + j;
        const Pair above = ab[u], below = xs[u];
        const T d = dg[u];
#pragma unroll
        for (int i = 0; i < 16 / (int)sizeof(IO); ++i) {
            const bool left = w + i < u;
            const Pair e = (left ? ab : xs)[w + i], f = left ? below : above;
            T v = fma_(f.x, e.x, f.s * e.s);
            if (w + i == u) v += d;
            q[i] = (IO)v;
        }
    });
    bool any = false;
    for (int q = tid; q < npts; q += kThreads) any |= flag[q] != 0;
    if (__syncthreads_or(any))
        for (int q = 0; q < npts; ++q)
            if (flag[q])
                ack_dense_rows<T, IO>(x + (size_t)q * n, static_cast<IO *>(a.out) + (size_t)(p0 + q) * n * n, n,
                                      split > 1 ? r0 : 0, split > 1 ? r1 : n);
}

// Fletcher-Powell, first launch: the diagonal's curvature 2 sum_m r_m P_ml
// (FP64 residuals), written to the diagonal of H.  For 3 <= n <= kGramSmall it
// also leaves sin x_l and cos x_l beside it, at columns l + 1 and l + 2 (mod
// n), where the second launch reads them before it overwrites H: FP64 sin and
// cos again would take that launch as long as its products.  One variable in
// compensated FP32 (T double, IO float): the whole entry 2 J^2 + curvature,
// whose terms can cancel, is formed here in FP64, rounded once, and there is no
// second launch.
constexpr int kGramSmall = 64;
__device__ __forceinline__ int beside(int l, int k, int n) { return l + k < n ? l + k : l + k - n; }
template <typename T, typename IO, bool kWide>
__global__ void __launch_bounds__(kFpThreads) fp_curvature_kernel(const StructArgs a, const FpShape sh, int ppb)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n;
    const long long p0 = (long long)blockIdx.x * ppb;
    const int P = (int)min((long long)ppb, a.batch - p0);
    FpTile<T, IO, false> tile(FpArgs{a.A, a.B, a.E, a.ld}, static_cast<const IO *>(a.x), nullptr, smem_raw, sh, P,
                              P * n);
    for (int q = threadIdx.x; q <= P; q += kFpThreads) {
        tile.base[q] = q * n;
        if (q < P) {
            tile.ns[q] = n;
            tile.xoff[q] = (p0 + q) * n;
            tile.eoff[q] = 0;
        }
    }
    __syncthreads();
    FpSums<T, 1> sums[kFpNpt];
    tile.template run<kWide>(0, n, sums);
    if constexpr (!std::is_same<T, IO>::value) {
        IO *H = static_cast<IO *>(a.out) + p0;
        bool bad = false;
#pragma unroll
        for (int i = 0; i < kFpNpt; ++i) {
            const int u = threadIdx.x + i * kFpThreads;
            if (u >= P) break;
            const T j = fp_jacobian<T>(a.A[0], a.B[0], tile.z[u].x, tile.z[u].y);
            const IO h = (IO)fma_(T(2) * j, j, tile.curvature(u, sums[i]));
            bad |= not_finite(h);
            H[u] = h;
        }
        if (__syncthreads_or(bad))
            for (int q = 0; q < P; ++q)
                if (not_finite(H[q]))
                    fp_dense_hessian<T, IO>(FpArgs{a.A, a.B, a.E, a.ld}, static_cast<const IO *>(a.x) + p0 + q, H + q,
                                            1, tile.z, tile.rd);
        return;
    }
    bool bad[kFpNpt] = {};
#pragma unroll
    for (int i = 0; i < kFpNpt; ++i) {
        const int u = threadIdx.x + i * kFpThreads;
        if (u >= P * n) break;
        const int l = u - tile.base[tile.qs[u]];
        IO *row = static_cast<IO *>(a.out) + ((size_t)p0 * n + u) * n;
        const T h = tile.curvature(u, sums[i]);
        bad[i] = not_finite(h);
        row[l] = (IO)h;
        if (n >= 3 && n <= kGramSmall) {
            row[beside(l, 1, n)] = (IO)narrow<T>(tile.z[u].x);
            row[beside(l, 2, n)] = (IO)narrow<T>(tile.z[u].y);
        }
    }
    // n > kGramSmall: the third launch looks at a point's first entry
    if (n > kGramSmall && __syncthreads_or(bad[0] || bad[1])) {
#pragma unroll
        for (int i = 0; i < kFpNpt; ++i)
            if (bad[i])
                static_cast<IO *>(a.out)[(size_t)(p0 + tile.qs[threadIdx.x + i * kFpThreads]) * n * n] =
                    nan_of(IO(0));
    }
}

// Second launch, n <= kGramSmall: ppc whole points per CTA, J in shared
// memory, one 4 x 4 block on or above the diagonal per thread; the result is
// staged in place of J and streamed out whole.
template <typename T, typename IO>
__global__ void __launch_bounds__(kThreads) fp_gram_small_kernel(const StructArgs a, int ppc, FastDiv fd)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n, nb = (n + 3) / 4, np = 4 * nb, nt = nb * (nb + 1) / 2, tid = threadIdx.x;
    const long long p0 = (long long)blockIdx.x * ppc;
    const int npts = (int)min((long long)ppc, a.batch - p0), nv = npts * n;
    Two<double> *z = reinterpret_cast<Two<double> *>(smem_raw);  // dense propagation only
    Two<T> *r = reinterpret_cast<Two<T> *>(z + n);
    T *J = reinterpret_cast<T *>(smem_raw + align_up((size_t)n * (sizeof(Two<double>) + sizeof(Two<T>)), 16));
    T *ts = J + (size_t)ppc * n * np, *tc = ts + ppc * n, *dg = tc + ppc * n;
    const IO *x = static_cast<const IO *>(a.x) + p0 * n;
    IO *H = static_cast<IO *>(a.out) + (size_t)p0 * n * n;
    bool bad = false;
    for (int u = tid; u < nv; u += kThreads) {
        const int l = u - fd.div(u) * n;
        const IO *row = H + (size_t)u * n;
        if (n >= 3) {
            ts[u] = (T)row[beside(l, 1, n)];
            tc[u] = (T)row[beside(l, 2, n)];
        } else {
            double s, c;
            sincos((double)x[u], &s, &c);
            ts[u] = (T)s;
            tc[u] = (T)c;
        }
        dg[u] = (T)row[l];
        bad |= not_finite(dg[u]);
    }
    __syncthreads();
    for (int e = tid; e < n * np; e += kThreads) {
        const int m = e / np, j = e - m * np;
        T av = T(0), bv = T(0);
        if (j < n) {
            av = narrow<T>(__ldg(&a.A[(size_t)m * a.ld + j]));
            bv = narrow<T>(__ldg(&a.B[(size_t)m * a.ld + j]));
        }
        for (int q = 0; q < npts; ++q)
            J[(size_t)q * n * np + e] = j < n ? fp_jacobian(av, bv, ts[q * n + j], tc[q * n + j]) : T(0);
    }
    __syncthreads();
    // the thread's point and block (bi <= bj), blocks of a point row by row
    const int q = tid / nt;
    int bi = 0, bj = tid - q * nt;
    while (bi < nb && bj >= nb - bi) {
        bj -= nb - bi;
        ++bi;
    }
    bj += bi;
    Gram4<T> g;
    g.init();
    if (q < npts) {
        const T *Jq = J + (size_t)q * n * np;
        int blk = 0;
        for (int m = 0; m < n; ++m) {
            g.add(Jq + m * np + 4 * bi, Jq + m * np + 4 * bj);
            if (++blk == kSumBlock) {
                g.flush();
                blk = 0;
            }
        }
        g.flush();
    }
    __syncthreads();
    if (q < npts) {
        T *Hs = J + (size_t)q * n * np;  // row stride np
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int ri = 4 * bi + i, rj = 4 * bj + j;
                if (ri >= n || rj >= n) continue;
                T v = g.value(i, j);
                if (ri == rj) v += dg[q * n + ri];
                Hs[ri * np + rj] = v;
                if (bi != bj) Hs[rj * np + ri] = v;
            }
    }
    __syncthreads();
    stream_rows(
        H, nv, n, fd, [&](int row, int j) { return J[(size_t)row * np + j]; },
        [&](int row, int j, IO *q) {
            constexpr int V = 16 / (int)sizeof(IO);
            Two<T> p[V / 2];  // n even: np and j are too
#pragma unroll
            for (int i = 0; i < V / 2; ++i) p[i] = *reinterpret_cast<const Two<T> *>(J + (size_t)row * np + j + 2 * i);
#pragma unroll
            for (int i = 0; i < V / 2; ++i) {
                q[2 * i] = (IO)p[i].x;
                q[2 * i + 1] = (IO)p[i].y;
            }
        });
    if (__syncthreads_or(bad))
        for (int k = 0; k < npts; ++k) {
            bool b = false;
            for (int l = tid; l < n; l += kThreads) b |= not_finite(dg[k * n + l]);
            if (__syncthreads_or(b))
                fp_dense_hessian<T, IO>(FpArgs{a.A, a.B, a.E, a.ld}, x + (size_t)k * n, H + (size_t)k * n * n, n, z, r);
        }
}

// Second launch, n > kGramSmall: a CTA takes one 64 x 64 block (I <= J) of one
// point, J formed for the two column ranges in tiles of kGramRows rows.
constexpr int kGramTile = 64;
constexpr int kGramRows = 16;
template <typename T>
__host__ __device__ constexpr size_t gram_smem()
{
    // two J tiles, the staged block, sin and cos of both ranges
    return (size_t)(2 * kGramRows * kGramTile + kGramTile * (kGramTile + 1) + 4 * kGramTile) * sizeof(T);
}
template <typename T, typename IO>
__global__ void __launch_bounds__(kThreads) fp_gram_kernel(const StructArgs a, int nbk)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *JI = reinterpret_cast<T *>(smem_raw), *JJ = JI + kGramRows * kGramTile;
    T *tile = JJ + kGramRows * kGramTile, *ts = tile + kGramTile * (kGramTile + 1), *tc = ts + 2 * kGramTile;
    const int n = a.n, tid = threadIdx.x, nt = nbk * (nbk + 1) / 2;
    const long long p = blockIdx.x / nt;
    int bi = 0, bj = (int)(blockIdx.x % nt);
    while (bj >= nbk - bi) {
        bj -= nbk - bi;
        ++bi;
    }
    bj += bi;
    const int i0 = bi * kGramTile, j0 = bj * kGramTile;
    const IO *x = static_cast<const IO *>(a.x) + p * n;
    IO *H = static_cast<IO *>(a.out) + (size_t)p * n * n;
    if (tid < 2 * kGramTile) {
        const int col = tid < kGramTile ? i0 + tid : j0 + tid - kGramTile;
        double s = 0.0, c = 0.0;
        if (col < n) sincos_rad(sincos_k(0), (double)x[col], s, c);
        ts[tid] = (T)s;
        tc[tid] = (T)c;
    }
    const int ty = tid / 16, tx = tid % 16;
    Gram4<T> g;
    g.init();
    for (int mb = 0; mb < n; mb += kGramRows) {
        __syncthreads();
        for (int e = tid; e < 2 * kGramRows * kGramTile; e += kThreads) {
            const int half = e / (kGramRows * kGramTile), w = e % (kGramRows * kGramTile);
            if (half && bi == bj) break;
            const int m = mb + w / kGramTile, k = w % kGramTile, col = (half ? j0 : i0) + k;
            T v = T(0);
            if (m < n && col < n)
                v = fp_jacobian(narrow<T>(__ldg(&a.A[(size_t)m * a.ld + col])),
                                narrow<T>(__ldg(&a.B[(size_t)m * a.ld + col])), ts[half * kGramTile + k],
                                tc[half * kGramTile + k]);
            (half ? JJ : JI)[w] = v;
        }
        __syncthreads();
        const T *Q = bi == bj ? JI : JJ;
#pragma unroll
        for (int m = 0; m < kGramRows; ++m) {
            g.add(JI + m * kGramTile + 4 * ty, Q + m * kGramTile + 4 * tx);
            if (m % kSumBlock == kSumBlock - 1) g.flush();
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int ri = 4 * ty + i, rj = 4 * tx + j;
            T v = g.value(i, j);
            if (bi == bj && ri == rj && i0 + ri < n) v += (T)H[(size_t)(i0 + ri) * n + i0 + ri];
            tile[ri * (kGramTile + 1) + rj] = v;
        }
    __syncthreads();
    for (int e = tid; e < kGramTile * kGramTile; e += kThreads) {
        const int u = e / kGramTile, w = e % kGramTile;
        if (i0 + u < n && j0 + w < n) H[(size_t)(i0 + u) * n + j0 + w] = (IO)tile[u * (kGramTile + 1) + w];
        if (bi != bj && j0 + u < n && i0 + w < n) H[(size_t)(j0 + u) * n + i0 + w] = (IO)tile[w * (kGramTile + 1) + u];
    }
}

// Third launch, n > kGramSmall: points with a curvature that is not finite (the
// first launch made their first entry NaN) by the dense propagation.
template <typename T, typename IO>
__global__ void __launch_bounds__(kThreads) fp_hessian_fix_kernel(const StructArgs a)
{
    __shared__ Two<double> z[kMaxVars];
    __shared__ Two<T> r[kMaxVars];
    __shared__ bool todo[kThreads];
    const size_t nn = (size_t)a.n * a.n;
    const long long p0 = (long long)blockIdx.x * kThreads, p = p0 + threadIdx.x;
    IO *H = static_cast<IO *>(a.out);
    todo[threadIdx.x] = p < a.batch && not_finite((T)H[(size_t)p * nn]);
    if (!__syncthreads_or(todo[threadIdx.x])) return;
    for (int k = 0; k < kThreads; ++k)
        if (todo[k])
            fp_dense_hessian<T, IO>(FpArgs{a.A, a.B, a.E, a.ld}, static_cast<const IO *>(a.x) + (p0 + k) * a.n,
                                    H + (size_t)(p0 + k) * nn, a.n, z, r);
}

template <typename T, typename IO>
cudaError_t ack_launch(const StructArgs &a, int G, unsigned blocks, cudaStream_t s)
{
    const int it = (a.n + G - 1) / G;
    const AckConst nc = ack_const(a.n);
    if constexpr (std::is_same<T, float>::value) {
        // whole 16-byte pieces per lane (a quarter of the load, store and
        // predicate instructions of a kernel bound by instruction issue:
        // n = 64, 524288 points, 143 -> 119 us with AckSums' halved merges)
        const size_t bits = (size_t)a.x | (size_t)a.v | (size_t)a.out;
        if (it > 2 && a.n % 4 == 0 && bits % 16 == 0) {
            if (it <= 4) ack_hvp_kernel<T, IO, 4, true><<<blocks, kAckThreads, 0, s>>>(a, G, nc);
            else if (it <= 8) ack_hvp_kernel<T, IO, 8, true><<<blocks, kAckThreads, 0, s>>>(a, G, nc);
            else ack_hvp_kernel<T, IO, 16, true><<<blocks, kAckThreads, 0, s>>>(a, G, nc);
            return cudaGetLastError();
        }
    }
    if (it <= 1) ack_hvp_kernel<T, IO, 1><<<blocks, kAckThreads, 0, s>>>(a, G, nc);
    else if (it <= 2) ack_hvp_kernel<T, IO, 2><<<blocks, kAckThreads, 0, s>>>(a, G, nc);
    else if (it <= 4) ack_hvp_kernel<T, IO, 4><<<blocks, kAckThreads, 0, s>>>(a, G, nc);
    else if (it <= 8) ack_hvp_kernel<T, IO, 8><<<blocks, kAckThreads, 0, s>>>(a, G, nc);
    else ack_hvp_kernel<T, IO, 16><<<blocks, kAckThreads, 0, s>>>(a, G, nc);
    return cudaGetLastError();
}

// Points per CTA of an FpTile kernel: at most as many pairs as its threads
// hold, and such that the last round of CTAs leaves few SMs idle (the FP64 pipe
// of an SM is the bound, 2 FMAs a clock, so the time is that of the SM with
// most work).  fmas: FP64 FMAs per (m, j).  A CTA's own cost, what the load of
// A and B and the barriers are not hidden by, is taken as 600 + n^2 / 10
// clocks.  Fewer than 128 pairs leave half of its threads without one.
int fp_points(int n, long long batch, int fmas)
{
    const int most = std::max(1, std::min(kFpMaxPts, kFpPairs / n));
    const double point = 0.5 * fmas * n * n + 10.0 * n, cta = 600.0 + 0.1 * n * n;
    int best = most;
    double best_cost = 1e300;
    for (int p = std::min(most, (127 + n) / n); p <= most; ++p) {
        const long long ctas = (batch + p - 1) / p, rounds = (ctas + kSms - 1) / kSms;
        const double cost = (double)rounds * (std::min<long long>(p, batch) * point + cta);
        if (cost <= best_cost) {
            best_cost = cost;
            best = p;
        }
    }
    return best;
}

template <typename T, typename IO, bool kHvp, bool kWide>
cudaError_t fp_launch_as(const StructArgs &a, cudaStream_t s)
{
    const int ppb = fp_points(a.n, a.batch, sizeof(T) == 8 ? (kHvp ? 8 : 4) : 2);
    const FpShape sh = fp_shape(a.n, a.n, ppb, ppb * a.n, sizeof(T) == 8);
    const size_t bytes = fp_smem<T>(sh).total;
    const long long blocks = (a.batch + ppb - 1) / ppb;
    if (blocks > kMaxBlocks) return cudaErrorInvalidConfiguration;
    auto kern = kHvp ? fp_hvp_kernel<T, IO, kWide> : fp_curvature_kernel<T, IO, kWide>;
    static std::atomic<int> configured[64];
    const cudaError_t e = opt_in_smem(kern, bytes, configured);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)blocks, kFpThreads, bytes, s>>>(a, sh, ppb);
    return cudaGetLastError();
}

template <typename T, typename IO, bool kHvp>
cudaError_t fp_launch(const StructArgs &a, cudaStream_t s)
{
    return a.n >= kFpWide ? fp_launch_as<T, IO, kHvp, true>(a, s) : fp_launch_as<T, IO, kHvp, false>(a, s);
}

template <typename T, typename IO>
cudaError_t hvp(int fn, const StructArgs &a, cudaStream_t s)
{
    if (fn == FN_FP) return fp_launch<T, IO, true>(a, s);
    const int G = fn == FN_ROSENBROCK ? ros_lanes(a.n) : ack_lanes(a.n, a.batch, sizeof(T) == 8);
    const long long ppb = (fn == FN_ACKLEY ? kAckThreads : kThreads) / G, blocks = (a.batch + ppb - 1) / ppb;
    if (blocks > kMaxBlocks) return cudaErrorInvalidConfiguration;
    if (fn == FN_ACKLEY) return ack_launch<T, IO>(a, G, (unsigned)blocks, s);
    ros_hvp_kernel<T, IO><<<(unsigned)blocks, kThreads, 0, s>>>(a, G);
    return cudaGetLastError();
}

// Output elements per CTA of the streaming Hessian kernels: enough to hide a
// CTA's start, few enough for several CTAs per SM.
constexpr int kHessElems = 16384;

template <typename T, typename IO>
cudaError_t fp_hessian(const StructArgs &a, FastDiv fd, cudaStream_t s)
{
    const int n = a.n;
    const int nbk = (n + kGramTile - 1) / kGramTile, nt = nbk * (nbk + 1) / 2;
    if (n > kGramSmall && a.batch > kMaxBlocks / nt) return cudaErrorInvalidConfiguration;
    cudaError_t e = fp_launch<T, IO, false>(a, s);
    if (e != cudaSuccess || !std::is_same<T, IO>::value) return e;  // one variable: the entry is whole
    static std::atomic<int> small_smem[64], gram_attr[64];
    if (n <= kGramSmall) {
        const int nb = (n + 3) / 4, np = 4 * nb, tiles = nb * (nb + 1) / 2;
        // points per CTA: one 4 x 4 block per thread, at most 64 KiB of J
        const size_t per = (size_t)n * (np + 3) * sizeof(T);
        int ppc = std::max(1, std::min(kThreads / tiles, (int)(64 * 1024 / per)));
        ppc = (int)std::min<long long>(ppc, std::max<long long>(1, (a.batch + 2 * kSms - 1) / (2 * kSms)));
        const size_t bytes = align_up((size_t)n * (sizeof(Two<double>) + sizeof(Two<T>)), 16) + ppc * per;
        const long long blocks = (a.batch + ppc - 1) / ppc;
        if (blocks > kMaxBlocks) return cudaErrorInvalidConfiguration;
        auto kern = fp_gram_small_kernel<T, IO>;
        e = opt_in_smem(kern, bytes, small_smem);
        if (e != cudaSuccess) return e;
        kern<<<(unsigned)blocks, kThreads, bytes, s>>>(a, ppc, fd);
        return cudaGetLastError();
    }
    auto kern = fp_gram_kernel<T, IO>;
    e = opt_in_smem(kern, gram_smem<T>(), gram_attr);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)(a.batch * nt), kThreads, gram_smem<T>(), s>>>(a, nbk);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    fp_hessian_fix_kernel<T, IO><<<(unsigned)((a.batch + kThreads - 1) / kThreads), kThreads, 0, s>>>(a);
    return cudaGetLastError();
}

template <typename T, typename IO>
cudaError_t hessian(int fn, const StructArgs &a, cudaStream_t s)
{
    const int n = a.n;
    const FastDiv fd{n == 1 ? 0u : (unsigned)((1ull << 32) / (unsigned)n + 1)};
    if (fn == FN_FP) return fp_hessian<T, IO>(a, fd, s);
    if (fn == FN_ROSENBROCK) {
        const long long total = a.batch * n;
        int rows = std::max(1, std::min(1024, kHessElems / n));
        rows = (int)std::min<long long>(rows, std::max<long long>(8, total / (2 * kSms)));
        const long long blocks = (total + rows - 1) / rows;
        if (blocks > kMaxBlocks) return cudaErrorInvalidConfiguration;
        const size_t bytes = (size_t)rows * (3 * sizeof(T) + sizeof(short));
        ros_hessian_kernel<T, IO><<<(unsigned)blocks, kThreads, bytes, s>>>(a, rows, fd);
        return cudaGetLastError();
    }
    const int split = std::max(1, (n * n + kHessElems - 1) / kHessElems);
    int ppc = split > 1 ? 1 : std::max(1, std::min(512 / n, kHessElems / (n * n)));
    ppc = (int)std::min<long long>(ppc, std::max<long long>(1, (a.batch + 2 * kSms - 1) / (2 * kSms)));
    const long long ctas = (a.batch + ppc - 1) / ppc;
    if (ctas > kMaxBlocks / split) return cudaErrorInvalidConfiguration;
    const size_t bytes = align_up((size_t)ppc * n * 5 * sizeof(T), 16) + ppc * (2 * sizeof(double) + 4 * sizeof(T)) +
                         (ppc + (ppc & 1)) * sizeof(int);
    ack_hessian_kernel<T, IO><<<(unsigned)(ctas * split), kThreads, bytes, s>>>(a, ppc, split, fd, ack_const(n));
    return cudaGetLastError();
}

}  // namespace

cudaError_t structured_hvp(int fn, bool f64, const StructArgs &a, cudaStream_t stream)
{
    if (f64) return hvp<double, double>(fn, a, stream);
    return a.n == 1 ? hvp<double, float>(fn, a, stream) : hvp<float, float>(fn, a, stream);
}

cudaError_t structured_hessian(int fn, bool f64, const StructArgs &a, cudaStream_t stream)
{
    if (f64) return hessian<double, double>(fn, a, stream);
    return a.n == 1 ? hessian<double, float>(fn, a, stream) : hessian<float, float>(fn, a, stream);
}

}  // namespace chessfad
