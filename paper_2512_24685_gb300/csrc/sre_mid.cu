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
          uint64_t x_begin, long long n, int alpha, double *__restrict__ part, double *__restrict__ per_x) {
    static_assert(NB == 1 || NB == 2, "one or two blocks per shift");
    constexpr int N = kTileBits + NB;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2 *buf = reinterpret_cast<double2 *>(smem_raw);  // moves
    double2 *park = buf + kTileSlots;                       // block 0 of two
    __shared__ double red[kThreads / 32];
    __shared__ FxShared sh;
    const int tid = threadIdx.x;

    for (long long g = blockIdx.x; g < n; g += gridDim.x) {
        const long long sidx = psis ? g / shifts_per_state : 0;
        const double2 *psi = psis ? reinterpret_cast<const double2 *>(psis[sidx]) : psi0;
        const uint64_t x = x_begin + (uint64_t)(g - sidx * shifts_per_state);
        FxExp u[NB];
        cx_t<fx> v[16];
#pragma unroll
        for (int tp = 0; tp < NB; ++tp) {
            block_values<fx>(v, block_pair(psi, N, x, tp), tid);
            u[tp] = fx_tile<12>(v, buf, tid, sh);
            if (tp + 1 < NB) {
#pragma unroll
                for (int i = 0; i < 16; ++i) park[(i << 8) | tid] = Cx<fx>::to(v[i]);
            }
        }
        double s = 0.0;
        int k = u[0].c;
        if constexpr (NB == 2) {
            k = fx_units<1>(0, max(u[0].c, u[1].c), max(u[0].s, u[1].s) + 1).k[2];
            const int q0 = k - u[0].c, q1 = k - u[1].c;
            cx_t<fx> w[16];
            auto join = [&](auto shift) {
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const cx_t<fx> p = Cx<fx>::from(park[(i << 8) | tid]);
                    const cx_t<fx> a = make_longlong2(shift(p.x, q0), shift(p.y, q0));
                    const cx_t<fx> b = make_longlong2(shift(v[i].x, q1), shift(v[i].y, q1));
                    w[i] = Cx<fx>::sub(a, b);
                    v[i] = Cx<fx>::add(a, b);
                }
            };
            if (max(q0, q1) <= 8)
                join([](long long a, int q) { return fx_shift_few(a, q); });
            else
                join([](long long a, int q) { return fx_shift(a, q); });
            s = sum_order<fx>(w, alpha);
        }
        s += sum_order<fx>(v, alpha);
        const double units = block_sum(s, red);
        if (tid == 0) {
            const double tot = fx_scale(units, alpha, k);
            part[g] = tot;
            if (per_x) per_x[g] = tot;
        }
    }
}

template <int NB>
cudaError_t launch_mid_t(const void *psi, const void *const *psis, int nstates, long long sps, uint64_t x_begin,
                         int alpha, double *part, double *per_x, const DeviceInfo &dev, cudaStream_t st) {
    const size_t smem = ((size_t)kTileSlots + (size_t)(NB - 1) * kTile) * sizeof(double2);
    auto kern = k_mid<NB>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const long long n = sps * (long long)nstates;
    if (n <= 0) return cudaSuccess;
    const int grid = (int)std::min<long long>(n, (long long)dev.sms * (NB == 1 ? 2 : 1));
    kern<<<grid, kThreads, smem, st>>>(reinterpret_cast<const double2 *>(psi), psis, sps, x_begin, n, alpha, part,
                                       per_x);
    return cudaGetLastError();
}

}  // namespace

bool mid_applies(int N, int elem_bytes) { return elem_bytes == 16 && (N == 13 || N == 14); }

cudaError_t launch_mid(int N, const void *psi, const void *const *psis, int nstates, long long sps, uint64_t x_begin,
                       int alpha, double *part, double *per_x, const DeviceInfo &dev, cudaStream_t st) {
    return N == 13 ? launch_mid_t<1>(psi, psis, nstates, sps, x_begin, alpha, part, per_x, dev, st)
                   : launch_mid_t<2>(psi, psis, nstates, sps, x_begin, alpha, part, per_x, dev, st);
}

}  // namespace sre
