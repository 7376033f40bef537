// sre_two.h -- host side of the FP32 two-pass kernel (sre_two.cu).
#pragma once
#include <cuda_runtime.h>

#include "sre_internal.h"

namespace sre {

struct TwoLayout {
    int C_log, U_log, W_log, R;
    bool share;  // an item's shifts share factors (sre_two.cu)
    uint64_t x0;
    long long n_chunks;  // per state
};

bool two_applies(int N, int elem_bytes);
LargeCfg choose_two_cfg(const DeviceInfo &dev, const Workspace &ws, int N);
// Chunks of one state over the shifts [xb, xe).
TwoLayout two_layout(const Workspace &ws, const LargeCfg &c, int N, uint64_t xb, uint64_t xe);
// Enqueue the sums over [xb, xe) of one state (psi) or of nstates states of a
// class (psis, device array): one partial per chunk in chunk_sum, state after
// state.  counters: three arrays of n_chunks words, counter_stride apart,
// zeroed by the caller; *work zeroed too.
cudaError_t launch_two(const Workspace &ws, const LargeCfg &c, int N, const void *psi, const void *const *psis,
                       int nstates, uint64_t xb, uint64_t xe, int alpha, double *chunk_sum, unsigned *counters,
                       size_t counter_stride, size_t counter_cap, unsigned long long *work, double *per_x,
                       long long wait_ns, cudaStream_t st);

}  // namespace sre
