// sre_mid.cu -- FP64 single-pass kernel (fixed-point transform, sre_tile.cuh)
// for N = 13 and 14: the halved transform of a shift is one or two 4096-entry
// blocks and stays inside one CTA.
//
// A CTA takes whole shifts, grid-strided over (state, shift): it forms the
// XOR-shifted products of each block, applies the 12-bit tile transform (bits
// 8-11 first), parks the first of two blocks in shared memory at positions
// only its own thread reads back (i << 8 | tid, no bank conflicts), then applies
// the butterfly across the blocks (transform bit 12).  The sum of powers is
// taken per thread and across the CTA in FP64 in a fixed tree: one partial per
// shift, the same in a single or a batched launch.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "sre_internal.h"
#include "sre_tile.cuh"

namespace sre {
using namespace dev;

namespace {

template <int NB>
__global__ void __launch_bounds__(kThreads, NB == 1 ? 2 : 1)
    k_mid(const double2 *__restrict__ psi0, const void *const *__restrict__ psis, long long shifts_per_state,
          uint64_t x_begin, long long n, int alpha, double *__restrict__ part, double *__restrict__ per_x,
          const int2 *__restrict__ fx_bn, const int *__restrict__ fx_e) {
    static_assert(NB == 1 || NB == 2, "one or two blocks per shift");
    constexpr int N = kTileBits + NB;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2 *buf = reinterpret_cast<double2 *>(smem_raw);  // moves
    double2 *park = buf + kTileSlots;                       // block 0 of two
    __shared__ double red[kThreads / 32];
    const int tid = threadIdx.x;

    for (long long g = blockIdx.x; g < n; g += gridDim.x) {
        const long long sidx = psis ? g / shifts_per_state : 0;
        const double2 *psi = psis ? reinterpret_cast<const double2 *>(psis[sidx]) : psi0;
        const uint64_t x = x_begin + (uint64_t)(g - sidx * shifts_per_state);
        // block bounds of the state and the unit's exponent of the shift
        const int2 *bn = fx_bn + (sidx << NB);
        const int k = fx_e[(sidx << NB) + (long long)(x >> kTileBits)];
        cx_t<fx> v[16];
#pragma unroll
        for (int tp = 0; tp < NB; ++tp) {
            const FxUnits un = fx_units(fx_bound(bn, 1 << NB, x, tp), k);
            block_values<fx>(v, block_pair(psi, N, x, tp), tid, un.a);
            fx_tile<12>(v, buf, tid, un);
            fx_rescale(v, k - un.c);
            if (tp + 1 < NB) {
#pragma unroll
                for (int i = 0; i < 16; ++i) park[(i << 8) | tid] = Cx<fx>::to(v[i]);
            }
        }
        double s = 0.0;
        if constexpr (NB == 2) {
            cx_t<fx> w[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const cx_t<fx> a = Cx<fx>::from(park[(i << 8) | tid]);
                w[i] = Cx<fx>::sub(a, v[i]);
                v[i] = Cx<fx>::add(a, v[i]);
            }
            s = sum_order<fx>(w, alpha);
        }
        s += sum_order<fx>(v, alpha);
        const double units = block_sum(s, red);
        if (tid == 0) {
            const double tot = half_scale<fx>(units, alpha, k);
            part[g] = tot;
            if (per_x) per_x[g] = tot;
        }
    }
}

template <int NB>
cudaError_t launch_mid_t(const void *psi, const void *const *psis, int nstates, long long sps, uint64_t x_begin,
                         int alpha, double *part, double *per_x, const int2 *fx_bn, const int *fx_e, const DeviceInfo &dev,
                         cudaStream_t st) {
    const size_t smem = ((size_t)kTileSlots + (size_t)(NB - 1) * kTile) * sizeof(double2);
    auto kern = k_mid<NB>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const long long n = sps * (long long)nstates;
    if (n <= 0) return cudaSuccess;
    const int grid = (int)std::min<long long>(n, (long long)dev.sms * (NB == 1 ? 2 : 1));
    kern<<<grid, kThreads, smem, st>>>(reinterpret_cast<const double2 *>(psi), psis, sps, x_begin, n, alpha, part,
                                       per_x, fx_bn, fx_e);
    return cudaGetLastError();
}

}  // namespace

bool mid_applies(int N, int elem_bytes) { return elem_bytes == 16 && (N == 13 || N == 14); }

cudaError_t launch_mid(int N, const void *psi, const void *const *psis, int nstates, long long sps, uint64_t x_begin,
                       int alpha, double *part, double *per_x, const int2 *fx_bn, const int *fx_e, const DeviceInfo &dev,
                       cudaStream_t st) {
    return N == 13 ? launch_mid_t<1>(psi, psis, nstates, sps, x_begin, alpha, part, per_x, fx_bn, fx_e, dev, st)
                   : launch_mid_t<2>(psi, psis, nstates, sps, x_begin, alpha, part, per_x, fx_bn, fx_e, dev, st);
}

}  // namespace sre
