// structured_tune.h -- host-side shapes of the structured kernels, shared by
// the contiguous launches (structured.cu) and the uneven-batch plan
// (ragged_structured.cu).
#pragma once

#include <algorithm>

#include "structured.cuh"
#include "structured.h"

namespace chessfad {

inline int pow2_ceil(int v)
{
    int p = 1;
    while (p < v) p <<= 1;
    return p;
}

// Lanes per point of the Rosenbrock kernel: about four variables per lane
// (independent loads in flight), at least 8 lanes where n has them (a warp's
// loads then cover whole 32-byte sectors).
inline int ros_lanes(int n)
{
    return std::min(32, std::max(pow2_ceil((n + 3) / 4), std::min(8, pow2_ceil(n))));
}

// Lanes per point of the Ackley kernel.  Each lane pays for the cross-lane
// sums and the tail's scalar functions about as much as for `over` variables,
// so few lanes with many variables each (at most 16) do least work; a batch
// too small to fill the GPU that way takes more lanes.
inline int ack_lanes(int n, long long batch, bool f64)
{
    const double over = f64 ? 2.0 : 1.0;
    int best = 1;
    double best_cost = 1e300;
    for (int g = 1; g <= 32; g <<= 1) {
        const int it = (n + g - 1) / g;
        if (it > 16 || (g > 1 && g >= 2 * n) || (!f64 && g < 8 && it > 1)) continue;
        const double waves = std::max(1.0, (double)batch * g / (kSms * 512.0));
        const double cost = (it + over) * waves;
        if (cost < best_cost) {
            best_cost = cost;
            best = g;
        }
    }
    return best;
}

// From this n on (at most 4 points per CTA) the rows of A and B are read from
// L2 instead of through a shared-memory tile: the tile would hold a few rows
// only, too few items for the CTA's warps between two barriers.  Time from L2
// over time with tiles, FP64 / FP32-comp: H v of 1000 points, n = 64 1.55/1.62,
// 96 1.21/1.49, 112 1.16/1.21, 127 1.00/0.91, 128 0.76/0.53, 160 0.77/0.49, 256
// 0.68/0.51, 512 0.79/0.41; of 16 points, 96 1.07/1.12, 127 0.79/0.65, 160
// 0.75/0.48; Hessians (curvature) between 0.97 and 1.16 up to n = 257, 0.98/0.73
// at 512; 200 uneven requests of sizes about n, 112 1.13/1.33, 128 1.02/1.05, 160
// 1.12/1.11, 200 0.97/1.10, 256 0.78/0.72, 512 0.74/0.44.
constexpr int kFpWide = 128;

// The shape of an FpTile: rows rows of A and B for P points, pairs pairs; f64:
// FP64 arithmetic.  All rows in one buffer within 48 KiB, else even parts of
// them in two buffers (two or more CTAs per SM).
inline FpShape fp_shape(int nmax, int rows, int P, int pairs, bool f64)
{
    const size_t row = (size_t)fp_stride(nmax) * (2 * sizeof(double) + (f64 ? 0 : 2 * sizeof(float)));
    FpShape s;
    s.nmax = nmax;
    s.pairs = pairs;
    s.bufs = 1;
    s.mt = rows;
    if (nmax >= kFpWide) {
        // rows per barrier: the CTA's warps' items, 4 per warp (fewer FP64
        // additions across lanes) while the rounded rows fit 64 KiB
        s.bufs = 0;
        s.lanes = nmax <= 256 ? 4 : 2;
        s.mt = kFpThreads / 32 * s.lanes / P;
        return s;
    }
    if ((size_t)rows * row > 48 * 1024) {
        const int most = std::max(1, (int)(40 * 1024 / row));
        const int tiles = (rows + most - 1) / most;
        s.bufs = 2;
        s.mt = (rows + tiles - 1) / tiles;
    }
    // pass 1: enough lanes per (point, row) to occupy the CTA's threads
    s.lanes = 1;
    while (s.lanes < 32 && s.lanes < nmax && P * s.mt * s.lanes < kFpThreads) s.lanes <<= 1;
    return s;
}

}  // namespace chessfad
