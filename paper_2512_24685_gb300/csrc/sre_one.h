// sre_one.h -- host side of the FP32 single-pass kernel (sre_one.cu).
#pragma once
#include <cuda_runtime.h>

#include "sre_internal.h"

namespace sre {

// Does it take N (FP32: elem_bytes 8)?  All shifts, one partial per shift.
bool one_applies(int N, int elem_bytes);
// Sums over [xb, xe) of one state (psi) or of nstates states (psis, device
// array): part[state * (xe - xb) + x - xb], also per_x if given (one state).
// *work: zeroed by the caller.
cudaError_t launch_one(int N, const void *psi, const void *const *psis, int nstates, uint64_t xb, uint64_t xe,
                       int alpha, double *part, double *per_x, unsigned long long *work, int *status,
                       long long wait_ns, const DeviceInfo &dev, cudaStream_t st);

}  // namespace sre
