// ragged_structured.cu -- the uneven batch by the structured evaluation
// (structured.cuh): the plan's tiles and the persistent kernel that takes them
// from a queue counter.
//
// Rosenbrock and Ackley requests are grouped by size, so that a tile's
// requests take the same number of lanes each.  Fletcher-Powell tiles pack
// points of similar size into the (point, variable) pairs of a CTA; a tile
// whose FP64 work would outlast the rest of the batch is cut by residual rows
// into parts.  Each part writes its partial sums (FP64) to slots of its own
// and counts itself; the part that completes the tile adds the slots in part
// order, so results do not depend on the order in which tiles run, and no CTA
// waits for another.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <numeric>

#include "structured.h"
#include "structured_tune.h"

namespace chessfad {
namespace {

constexpr int kThreads = kFpThreads;

// 4000 requests, n log-uniform in 2 .. 512, compensated FP32: dense 308 ms, here
// 0.258 ms.  The FP64 FMAs of the residuals, nearly all of them in the
// Fletcher-Powell requests of n >= 128, need 0.106 ms; the rest is the latency
// of the large requests' parts (one part alone takes 55 us, 16 of them FP64).

// The tile functions are calls, so that each has registers of its own: inlined
// into one kernel, the FP64 and many-variable variants made all of them spill.
template <typename T, typename IO>
__device__ __noinline__ void lanes_tile(const SRaggedArgs &a, const STile &t)
{
    const IO *x = static_cast<const IO *>(a.x), *v = static_cast<const IO *>(a.v);
    IO *out = static_cast<IO *>(a.out);
    const int G = t.lanes, groups = kThreads / G, lane = threadIdx.x & (G - 1);
    for (int k = 0; k < t.count; k += groups) {  // uniform in the CTA (shuffles)
        const int r = k + (int)threadIdx.x / G;
        const bool active = r < t.count;
        const int e = t.first + (active ? r : 0), n = a.n[e];
        const long long o = a.off[e];
        if (t.fn == FN_ROSENBROCK) {
            ros_point<T, IO>(x + o, v + o, out + o, n, lane, G, active, false);
        } else {
            const AckConst nc = ack_const(n);
            if constexpr (!std::is_same<T, IO>::value) {  // one variable
                ack_point<T, IO, 1>(x + o, v + o, out + o, n, lane, G, active, false, nc);
                continue;
            }
            switch (t.epl) {
            case 1: ack_point<T, IO, 1>(x + o, v + o, out + o, n, lane, G, active, false, nc); break;
            case 4: ack_point<T, IO, 4>(x + o, v + o, out + o, n, lane, G, active, false, nc); break;
            case 8: ack_point<T, IO, 8>(x + o, v + o, out + o, n, lane, G, active, false, nc); break;
            default: ack_point<T, IO, 16>(x + o, v + o, out + o, n, lane, G, active, false, nc); break;
            }
        }
    }
}

template <typename T, typename IO, bool kWide>
__device__ __noinline__ void fp_ragged_tile(const SRaggedArgs &a, const STile &t, unsigned char *smem)
{
    __shared__ int s_last;
    IO *out = static_cast<IO *>(a.out);
    const FpShape sh{t.nmax, t.mt, t.bufs, t.pairs, t.lanes};
    FpTile<T, IO, true> tile(FpArgs{a.A, a.B, a.Epack, a.ld}, static_cast<const IO *>(a.x),
                             static_cast<const IO *>(a.v), smem, sh, t.count, t.pairs);
    for (int q = threadIdx.x; q <= t.count; q += kThreads) {
        const int e = t.first + q;
        if (q < t.count) {
            tile.ns[q] = a.n[e];
            tile.base[q] = a.base[e];
            tile.xoff[q] = a.off[e];
            tile.eoff[q] = a.eoff[e];
        } else {
            tile.base[q] = t.pairs;
        }
    }
    __syncthreads();
    FpSums<T, 2> sums[kFpNpt];
    tile.template run<kWide>(t.m0, t.m1, sums);
    if (t.parts > 1) {
        double *slot = a.slots + t.slot + (long long)t.part * 4 * t.pairs;
#pragma unroll
        for (int i = 0; i < kFpNpt; ++i) {
            const int u = threadIdx.x + i * kThreads;
            if (u < t.pairs)
                for (int k = 0; k < 4; ++k) slot[k * t.pairs + u] = sums[i].wide(k);
        }
        // publish the slot, count the part; the last one adds them all
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) s_last = atomicAdd(&a.done[t.done], 1) + 1 == t.parts;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
    }
    bool bad = false;
#pragma unroll
    for (int i = 0; i < kFpNpt; ++i) {
        const int u = threadIdx.x + i * kThreads;
        if (u >= t.pairs) break;
        T f[4];
        if (t.parts > 1) {
            // every part's four sums, the loads of four parts in flight
            const double *slot = a.slots + t.slot + u;
            double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
            for (int p = 0; p < t.parts; ++p)
#pragma unroll
                for (int k = 0; k < 4; ++k) s[k] += __ldcg(slot + ((long long)p * 4 + k) * t.pairs);
#pragma unroll
            for (int k = 0; k < 4; ++k) f[k] = (T)s[k];
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) f[k] = sums[i].value(k);
        }
        const T o = tile.combine(u, f[0], f[1], f[2], f[3]);
        bad |= not_finite(o);
        out[tile.xoff[tile.qs[u]] + (u - tile.base[tile.qs[u]])] = (IO)o;
    }
    // the dense uneven batch adds the rows of n >= 128 in FP64
    if (__syncthreads_or(bad)) fp_dense_points<T, IO>(tile, out, 128);
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 2) structured_ragged_kernel(const __grid_constant__ SRaggedArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_tile;
    for (;;) {
        __syncthreads();  // the previous tile is done with shared memory and s_tile
        if (threadIdx.x == 0) s_tile = atomicAdd(a.counter, 1);
        __syncthreads();
        if (s_tile >= a.ntiles) break;
        const STile t = a.tiles[s_tile];
        if (IsComp<T>::value && t.f64) {
            if (t.fn == FN_FP) fp_ragged_tile<double, T, false>(a, t, smem_raw);
            else lanes_tile<double, T>(a, t);
        } else {
            if (t.fn == FN_FP && t.bufs == 0) fp_ragged_tile<T, T, true>(a, t, smem_raw);
            else if (t.fn == FN_FP) fp_ragged_tile<T, T, false>(a, t, smem_raw);
            else lanes_tile<T, T>(a, t);
        }
    }
}

}  // namespace

void structured_plan(const chessfad_request *reqs, long long nreq, int prec, SPlan &pl)
{
    const bool f64 = prec == CHESSFAD_FP64;
    // entries: by function, one-variable requests apart (in compensated FP32
    // they are computed in FP64), then by size, largest first
    std::vector<int> order(nreq);
    auto group = [&](int q) { return 2 * reqs[q].fn + (reqs[q].n == 1); };
    auto key = [&](long long q) { return group((int)q) * (kMaxVars + 1) + kMaxVars - reqs[q].n; };
    std::vector<long long> at(6 * (kMaxVars + 1) + 1, 0);  // counting sort: where each key starts
    for (long long q = 0; q < nreq; ++q) ++at[key(q) + 1];
    std::partial_sum(at.begin(), at.end(), at.begin());
    for (long long q = 0; q < nreq; ++q) order[at[key(q)]++] = (int)q;
    pl.n.resize(nreq);
    pl.off.resize(nreq);
    pl.eoff.resize(nreq);
    pl.base.assign(nreq, 0);
    for (long long e = 0; e < nreq; ++e) {
        const chessfad_request &r = reqs[order[e]];
        pl.n[e] = r.n;
        pl.off[e] = r.off;
        pl.eoff[e] = r.fn == CHESSFAD_FLETCHER_POWELL ? r.eoff : 0;
    }
    // FP64 FMAs of a point: the residuals, in FP64 all eight per (m, j), and
    // sin and cos
    auto fp_cost = [&](double n) { return n * n * (f64 ? 8.0 : 2.0) + 40.0 * n; };
    double total = 0.0;
    for (long long e = 0; e < nreq; ++e)
        total += reqs[order[e]].fn == CHESSFAD_FLETCHER_POWELL ? fp_cost(pl.n[e]) : (f64 ? 50.0 : 4.0) * pl.n[e];
    // a tile larger than this is split: about a quarter of an SM's share of
    // the batch, and at least 15 us of its FP64 pipe (2 FMAs a clock).  4000
    // requests up to n = 512: a sixteenth 268 us, an eighth 268, a quarter 257;
    // at least 7.5 us 258, 15 us 257, 30 us 256; one request of n = 505: 64, 65
    // and 85 us.
    const double most = std::max(62000.0, total / (kSms * 4.0));
    std::vector<std::pair<double, STile>> work;
    long long end = 0;  // of the current tile's group
    for (long long e = 0; e < nreq;) {
        const int fn = reqs[order[e]].fn, nmax = pl.n[e];
        if (e == end)
            while (end < nreq && group(order[end]) == group(order[e])) ++end;
        STile t{};
        t.fn = fn;
        t.first = (int)e;
        t.f64 = !f64 && nmax == 1;
        t.nmax = nmax;
        t.parts = 1;
        if (fn == CHESSFAD_FLETCHER_POWELL) {
            double cost = 0.0;
            while (e < end && t.count < kFpMaxPts && t.pairs + pl.n[e] <= kFpPairs && 5 * pl.n[e] + 20 >= 4 * nmax) {
                pl.base[e] = t.pairs;
                t.pairs += pl.n[e];
                cost += fp_cost(pl.n[e]);
                ++t.count;
                ++e;
            }
            t.parts = std::max(1, std::min((nmax + 15) / 16, (int)std::ceil(cost / most)));
            if (t.parts > 1) {
                t.done = pl.ndone++;
                t.slot = pl.slot_elems;
                pl.slot_elems += (long long)t.parts * 4 * t.pairs;
            }
            for (t.part = 0; t.part < t.parts; ++t.part) {
                t.m0 = nmax * t.part / t.parts;
                t.m1 = nmax * (t.part + 1) / t.parts;
                const bool wide = f64 || t.f64;
                const FpShape sh = fp_shape(nmax, t.m1 - t.m0, t.count, t.pairs, wide);
                t.mt = sh.mt;
                t.bufs = sh.bufs;
                t.lanes = sh.lanes;
                pl.smem = std::max(pl.smem, wide ? fp_smem<double>(sh).total : fp_smem<float>(sh).total);
                work.push_back({cost / t.parts + 40.0 * t.pairs, t});
            }
            continue;
        }
        t.lanes = fn == CHESSFAD_ROSENBROCK ? ros_lanes(nmax) : ack_lanes(nmax, end - e, f64 || t.f64);
        const int it = (nmax + t.lanes - 1) / t.lanes;
        t.epl = it <= 1 ? 1 : it <= 4 ? 4 : it <= 8 ? 8 : 16;
        // rounds of the CTA's lane groups: fewer when the batch is small
        const int groups = kThreads / t.lanes;
        const long long rounds = std::max<long long>(1, std::min<long long>(4, (end - e) / (4LL * kSms * groups)));
        double elems = 0.0;
        while (e < end && t.count < groups * rounds && 2 * pl.n[e] >= nmax) {
            elems += pl.n[e];
            ++t.count;
            ++e;
        }
        work.push_back({elems * (fn == CHESSFAD_ACKLEY ? (f64 ? 50.0 : 4.0) : (f64 ? 12.0 : 1.0)), t});
    }
    std::stable_sort(work.begin(), work.end(),
                     [](const std::pair<double, STile> &p, const std::pair<double, STile> &q) { return p.first > q.first; });
    for (const auto &w : work) pl.tiles.push_back(w.second);
    pl.smem = std::max<size_t>(pl.smem, 16);
}

namespace {
template <typename T>
cudaError_t grid_of(size_t smem, int *grid)
{
    auto kern = structured_ragged_kernel<T>;
    static std::atomic<int> configured[64];
    cudaError_t e = opt_in_smem(kern, smem, configured);
    int dev = 0, per_sm = 0, sms = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    *grid = std::max(1, per_sm) * sms;
    return e;
}
}  // namespace

cudaError_t structured_ragged_grid(bool f64, size_t smem, int *grid)
{
    return f64 ? grid_of<double>(smem, grid) : grid_of<float>(smem, grid);
}

cudaError_t structured_ragged(bool f64, const SRaggedArgs &a, size_t smem, int grid, cudaStream_t stream)
{
    const int blocks = std::min(grid, a.ntiles);
    if (f64) structured_ragged_kernel<double><<<blocks, kThreads, smem, stream>>>(a);
    else structured_ragged_kernel<float><<<blocks, kThreads, smem, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace chessfad
