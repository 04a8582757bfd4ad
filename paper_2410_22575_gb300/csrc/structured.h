// structured.h -- host-side entry points of the structured evaluation
// (structured.cuh): the library's own choice when a call names neither a
// chunk size nor a method.
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "../../include/chessfad.h"

namespace chessfad {

constexpr int kMaxVars = 512;  // CHESSFAD_MAX_N
// SMs of GB300, for the rules that share work out; plans are built on hosts
// without a device too, so it is a constant.  Results are right for any count.
constexpr int kSms = 152;

struct StructArgs {
    const void *x;
    const void *v;  // HVP only
    void *out;
    const double *A, *B, *E;  // Fletcher-Powell
    int ld;
    long long batch;
    int n;
    bool wide;  // compensated FP32: the dense HVP of this size adds its rows in FP64
};

// out = H v over a contiguous batch.  cudaErrorInvalidConfiguration when the
// batch needs more than one launch grid.  f64: FP64 data and arithmetic; else
// float data, computed in compensated FP32 (in FP64 at n = 1).
cudaError_t structured_hvp(int fn, bool f64, const StructArgs &a, cudaStream_t stream);

// out = every Hessian, as structured_hvp.
cudaError_t structured_hessian(int fn, bool f64, const StructArgs &a, cudaStream_t stream);

// ---- uneven batches (ragged_structured.cu)

// A CTA's unit of work: `count` requests of one function from entry `first` of
// the request tables.
struct STile {
    int fn, first, count;
    int f64;    // compensated FP32: one-variable requests, computed in FP64
    int lanes;  // Rosenbrock, Ackley: lanes per request; Fletcher-Powell: FpShape::lanes
    int epl;    // Ackley: variables per lane
    // Fletcher-Powell: the (point, variable) pairs, the shape, the rows of this
    // part, and, with several parts, the tile's counter and first slot element
    int pairs, nmax, mt, bufs, m0, m1, parts, part, done;
    long long slot;
};

struct SRaggedArgs {
    const void *x;
    const void *v;
    void *out;
    const double *A, *B, *Epack;
    int ld, ntiles;
    const STile *tiles;
    const long long *off, *eoff;  // per entry: element offsets of x, v, out and of E
    const int *n, *base;          // size; first pair in its tile
    int *counter, *done;          // the tile queue; parts completed per split tile
    double *slots;                // partial sums of split tiles
};

struct SPlan {
    std::vector<STile> tiles;
    std::vector<long long> off, eoff;
    std::vector<int> n, base;
    long long slot_elems = 0;
    int ndone = 0;
    size_t smem = 0;
};

// The tiles of the (validated) requests for precision prec, costly ones first.
void structured_plan(const chessfad_request *reqs, long long nreq, int prec, SPlan &plan);

// CTAs of the persistent grid on the current device (with the plan's shared
// memory, which this call makes available to the kernel), and the launch.
cudaError_t structured_ragged_grid(bool f64, size_t smem, int *grid);
cudaError_t structured_ragged(bool f64, const SRaggedArgs &a, size_t smem, int grid, cudaStream_t stream);

}  // namespace chessfad
