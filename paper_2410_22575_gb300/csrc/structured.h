// structured.h -- host-side entry points of the structured evaluation
// (structured.cuh): the library's own choice when a call names neither a
// chunk size nor a method.
#pragma once

#include <cuda_runtime.h>

namespace chessfad {

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

}  // namespace chessfad
