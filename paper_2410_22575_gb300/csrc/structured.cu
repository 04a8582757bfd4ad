// structured.cu -- kernels and launches of the structured evaluation over a
// contiguous batch (structured.cuh).
//
// H v through the default call, GB300, dense symmetric method -> here:
//   Ackley n = 64, FP64, 65536 points            102.2 ms -> 0.39 ms
//   Ackley n = 64, FP32-comp, 524288 points       15.9 ms -> 0.35 ms
//   Fletcher-Powell n = 32, FP32-comp, 16384       1.83 ms -> 0.100 ms
//   Fletcher-Powell n = 75, FP64, 1000            151.7 ms -> 0.119 ms
// The Rosenbrock kernel streams x and v; the other two are bound by the FP64
// pipe (sin, cos and the sums under sqrt and exp; the residuals), in
// compensated FP32 too.
#include <algorithm>
#include <atomic>

#include "structured.cuh"
#include "structured.h"

namespace chessfad {
namespace {

constexpr int kThreads = 256;
constexpr long long kMaxBlocks = 0x7fffffffLL;

int pow2_ceil(int v)
{
    int p = 1;
    while (p < v) p <<= 1;
    return p;
}

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

template <typename T, typename IO, int EPL>
__global__ void __launch_bounds__(kThreads) ack_hvp_kernel(const StructArgs a, int G, double inv_n)
{
    const long long p = ((long long)blockIdx.x * kThreads + threadIdx.x) / G;
    const int t = threadIdx.x & (G - 1);
    const bool active = p < a.batch;
    const size_t o = active ? (size_t)p * a.n : 0;
    ack_point<T, IO, EPL>(static_cast<const IO *>(a.x) + o, static_cast<const IO *>(a.v) + o,
                          static_cast<IO *>(a.out) + o, a.n, t, G, active, a.wide, inv_n);
}

template <typename T, typename IO>
__global__ void __launch_bounds__(kFpThreads) fp_hvp_kernel(const StructArgs a, const FpShape sh, int ppb)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n;
    const long long p0 = (long long)blockIdx.x * ppb;
    const int P = (int)min((long long)ppb, a.batch - p0);
    const FpArgs fa{a.A, a.B, a.E, a.ld};
    IO *out = static_cast<IO *>(a.out);
    FpTile<T, IO> tile(fa, static_cast<const IO *>(a.x), static_cast<const IO *>(a.v), smem_raw, sh, P, P * n);
    for (int q = threadIdx.x; q <= P; q += kFpThreads) {
        tile.base[q] = q * n;
        if (q < P) {
            tile.ns[q] = n;
            tile.xoff[q] = (p0 + q) * n;
            tile.eoff[q] = 0;
        }
    }
    __syncthreads();
    FpSums<T, 4> sums[kFpNpt];
    tile.run(0, n, sums);
    bool bad = false;
#pragma unroll
    for (int i = 0; i < kFpNpt; ++i) {
        const int u = threadIdx.x + i * kFpThreads;
        if (u >= P * n) break;
        const T o = tile.combine(u, sums[i].value(0), sums[i].value(1), sums[i].value(2), sums[i].value(3));
        bad |= not_finite(o);
        out[p0 * n + u] = (IO)o;
    }
    if (__syncthreads_or(bad)) fp_dense_points<T, IO>(tile, out, a.wide);
}

// Lanes per point of the Rosenbrock kernel: about four variables per lane
// (independent loads in flight), at least 8 lanes where n has them (a warp's
// loads then cover whole 32-byte sectors).
int ros_lanes(int n)
{
    return std::min(32, std::max(pow2_ceil((n + 3) / 4), std::min(8, pow2_ceil(n))));
}

// Lanes per point of the Ackley kernel.  Each lane pays for the cross-lane
// sums and the tail's scalar functions about as much as for `over` variables,
// so few lanes with many variables each (at most 16) do least work; a batch
// too small to fill the GPU that way takes more lanes.
int ack_lanes(int n, long long batch, bool f64)
{
    const double over = f64 ? 2.0 : 1.0;
    int best = 1;
    double best_cost = 1e300;
    for (int g = 1; g <= 32; g <<= 1) {
        const int it = (n + g - 1) / g;
        if (it > 16 || (g > 1 && g >= 2 * n)) continue;
        const double waves = std::max(1.0, (double)batch * g / (152.0 * 512.0));
        const double cost = (it + over) * waves;
        if (cost < best_cost) {
            best_cost = cost;
            best = g;
        }
    }
    return best;
}

template <typename T, typename IO>
cudaError_t ack_launch(const StructArgs &a, int G, unsigned blocks, cudaStream_t s)
{
    const int it = (a.n + G - 1) / G;
    const double inv_n = 1.0 / a.n;
    if (it <= 1) ack_hvp_kernel<T, IO, 1><<<blocks, kThreads, 0, s>>>(a, G, inv_n);
    else if (it <= 2) ack_hvp_kernel<T, IO, 2><<<blocks, kThreads, 0, s>>>(a, G, inv_n);
    else if (it <= 4) ack_hvp_kernel<T, IO, 4><<<blocks, kThreads, 0, s>>>(a, G, inv_n);
    else if (it <= 8) ack_hvp_kernel<T, IO, 8><<<blocks, kThreads, 0, s>>>(a, G, inv_n);
    else ack_hvp_kernel<T, IO, 16><<<blocks, kThreads, 0, s>>>(a, G, inv_n);
    return cudaGetLastError();
}

// Rows of A and B per tile: all of them within 64 KiB (two or more CTAs per
// SM hide the barriers between the passes), else even parts of the rows.
template <typename T>
FpShape fp_shape(int nmax, int rows, int P)
{
    const size_t row = (size_t)fp_stride(nmax) * 2 * (sizeof(double) + (sizeof(T) == 4 ? sizeof(float) : 0));
    const int most = std::max(1, (int)(64 * 1024 / row));
    const int tiles = (rows + most - 1) / most;
    FpShape s;
    s.nmax = nmax;
    s.mt = (rows + tiles - 1) / tiles;
    // pass 1: enough lanes per (point, row) to occupy the CTA's threads
    s.lanes = 1;
    while (s.lanes < 32 && s.lanes < nmax && P * s.mt * s.lanes < kFpThreads) s.lanes <<= 1;
    return s;
}

template <typename T, typename IO>
cudaError_t fp_launch(const StructArgs &a, cudaStream_t s)
{
    // Points per CTA: as many pairs as its threads hold, fewer when the batch
    // would leave SMs without a CTA.
    int ppb = std::max(1, std::min(kFpMaxPts, kFpPairs / a.n));
    ppb = (int)std::min<long long>(ppb, std::max<long long>(1, (a.batch + 303) / 304));
    const FpShape sh = fp_shape<T>(a.n, a.n, ppb);
    const size_t bytes = fp_smem<T>(sh.nmax, sh.mt).total;
    const long long blocks = (a.batch + ppb - 1) / ppb;
    if (blocks > kMaxBlocks) return cudaErrorInvalidConfiguration;
    auto kern = fp_hvp_kernel<T, IO>;
    static std::atomic<int> configured[64];
    const cudaError_t e = opt_in_smem(kern, bytes, configured);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)blocks, kFpThreads, bytes, s>>>(a, sh, ppb);
    return cudaGetLastError();
}

template <typename T, typename IO>
cudaError_t hvp(int fn, const StructArgs &a, cudaStream_t s)
{
    if (fn == FN_FP) return fp_launch<T, IO>(a, s);
    const int G = fn == FN_ROSENBROCK ? ros_lanes(a.n) : ack_lanes(a.n, a.batch, sizeof(T) == 8);
    const long long ppb = kThreads / G, blocks = (a.batch + ppb - 1) / ppb;
    if (blocks > kMaxBlocks) return cudaErrorInvalidConfiguration;
    if (fn == FN_ACKLEY) return ack_launch<T, IO>(a, G, (unsigned)blocks, s);
    ros_hvp_kernel<T, IO><<<(unsigned)blocks, kThreads, 0, s>>>(a, G);
    return cudaGetLastError();
}

}  // namespace

cudaError_t structured_hvp(int fn, bool f64, const StructArgs &a, cudaStream_t stream)
{
    if (f64) return hvp<double, double>(fn, a, stream);
    return a.n == 1 ? hvp<double, float>(fn, a, stream) : hvp<float, float>(fn, a, stream);
}

}  // namespace chessfad
