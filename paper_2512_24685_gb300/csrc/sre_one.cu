// sre_one.cu -- FP32 single-pass kernel for 13 <= N <= 16: the halved
// transform of a shift (N - 1 bits, sre_wht32.cuh) stays inside one CTA, so
// nothing goes through a scratch ring and no CTA waits for another.
//
// A CTA of 256 threads transforms blocks of 8192 entries (64 KB, 32 entries
// per thread).  N = 13: a block holds two shifts; N = 14: one; N = 15, 16: a
// shift is two or four blocks, all but the last parked: tensor memory takes
// one or two of them (a thread writes its 64 columns and reads them back, off
// the shared-memory pipe), shared memory the third of N = 16, beside a move
// buffer of half the size.  Two CTAs fit an SM in every case (128 registers).
//
// What bounds it: the shared-memory / L1 pipe and the FP32 pipe about evenly
// (per entry of the block one load of each factor, one move through shared
// memory, three shuffles; per 32 entries some 12 cycles of the L1 pipe and 10
// of the FP32 pipes), with 16 warps per SM to cover latency.  Measured on
// GB300, all shifts of one state: N = 16 4.6 ms (the two-pass kernel with 16
// entries per thread and full transforms below x = 4096: 9.9 ms), N = 15 1.24
// ms (2.04 ms, a CTA per SM parking three 4096-entry blocks in shared memory),
// N = 14 in a batch of 60 0.31 ms per state (0.45 ms); 20.6 SM cycles per 32
// complex entries at N = 16.
//
// Tiles (one block's shifts, or one shift) are claimed from one counter: the
// warps of an SM progress unevenly and a fixed split left some idle at the
// end (N = 16: 5.1 ms).  The claim travels through an mbarrier, a bounded wait
// like every other.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "sre_internal.h"
#include "sre_one.h"
#include "sre_wht32.cuh"

namespace sre {
using namespace dev;

namespace {

template <int N>
struct One {
    static constexpr int kBits = N - 1;                                    // transform bits of a shift (N < 14)
    static constexpr int kShifts = N < 14 ? 1 << (14 - N) : 1;             // shifts in one block
    static constexpr int kBlocks = N > 14 ? 1 << (N - 14) : 1;             // blocks of one shift
    // Parked blocks of a shift: tensor memory holds one (N = 15) or two (N =
    // 16) per thread, N = 16 a third in shared memory beside a move buffer of
    // half the size.
    static constexpr int kTmemBlocks = kBlocks == 1 ? 0 : kBlocks == 2 ? 1 : 2;
    static constexpr bool kHalfMove = kBlocks == 4;
    static constexpr size_t kSmem = kHalfMove ? kMoveBytes / 2 + 8192 * sizeof(float2) : kMoveBytes;
    // Doubled products below x = 4096 (fp32_doubled).  N = 16 doubles all shifts'
    // results instead, at orders above 4 alone: the branch in each of its four
    // transforms costs 3 % (4.64 -> 4.78 ms).
    static constexpr bool kTwice = N < 16;
    static constexpr uint32_t kCols = 64 * kTmemBlocks;  // tensor-memory columns of a warp
};

__device__ __forceinline__ void tmem_get4(uint32_t addr, c64_t (&v)[4]) {
    uint32_t r[8];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(addr)
        : "memory");
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = ((unsigned long long)r[2 * q + 1] << 32) | r[2 * q];
}

// The last transform bits of a shift, across its blocks (the last one in v,
// the others parked), and the sum of powers over all of them: FP32 over 16
// entries, FP64 above.
template <int N, int A>
__device__ __forceinline__ double one_blocks(const c64_t (&v)[32], uint32_t tmem, const c64_t *park, int tid,
                                             int alpha) {
    constexpr int kBlocks = One<N>::kBlocks;
    double s = 0.0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        c64_t acc[kBlocks];
#pragma unroll
        for (int m = 0; m < kBlocks; ++m) acc[m] = Cx<float>::zero();
#pragma unroll
        for (int i = 16 * h; i < 16 * h + 16; i += 4) {
            c64_t a0[4], a1[4];
            tmem_get4(tmem + 2 * i, a0);
            if constexpr (kBlocks == 4) tmem_get4(tmem + 64 + 2 * i, a1);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if constexpr (kBlocks == 2) {
                    acc[0] = w32_acc<A>(acc[0], Cx<float>::add(a0[q], v[i + q]), alpha);
                    acc[1] = w32_acc<A>(acc[1], Cx<float>::sub(a0[q], v[i + q]), alpha);
                } else {
                    const c64_t a2 = park[((i + q) << 8) | tid];
                    const c64_t b0 = Cx<float>::add(a0[q], a1[q]), b1 = Cx<float>::sub(a0[q], a1[q]);
                    const c64_t b2 = Cx<float>::add(a2, v[i + q]), b3 = Cx<float>::sub(a2, v[i + q]);
                    acc[0] = w32_acc<A>(acc[0], Cx<float>::add(b0, b2), alpha);
                    acc[1] = w32_acc<A>(acc[1], Cx<float>::add(b1, b3), alpha);
                    acc[2] = w32_acc<A>(acc[2], Cx<float>::sub(b0, b2), alpha);
                    acc[3] = w32_acc<A>(acc[3], Cx<float>::sub(b1, b3), alpha);
                }
            }
        }
#pragma unroll
        for (int m = 0; m < kBlocks; ++m) s += w32_flush(acc[m]);
    }
    return s;
}

// Bounded wait for the claim: on expiry SRE_ETIMEDOUT is recorded and the
// wait goes on (the claim is one atomic away), so that the CTA stays together
// and leaves at the next claim.
__device__ __forceinline__ void one_wait(uint32_t mbar, uint32_t parity, int *status, long long wait_ns) {
    if (mbar_test_wait(mbar, parity)) return;
    const unsigned long long t0 = globaltimer_ns();
    bool late = false;
    for (unsigned it = 0; it < (1u << 28); ++it) {
        if (mbar_test_wait(mbar, parity)) return;
        if (!late && (long long)(globaltimer_ns() - t0) > wait_ns) {
            late = true;
            atomicCAS(status, 0, (int)SRE_ETIMEDOUT);
        }
    }
}

template <int N>
__global__ void __launch_bounds__(kBlockThreads, 2)
    k_one(const float2 *__restrict__ psi0, const void *const *__restrict__ psis, long long tiles_per_state,
          uint64_t x_begin, uint64_t x_end, long long n_tiles, int alpha, double *__restrict__ part,
          double *__restrict__ per_x, unsigned long long *work, int *status, long long wait_ns) {
    using O = One<N>;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ double red[kBlockThreads / 32];
    __shared__ uint32_t s_tmem;
    __shared__ long long s_tile[2];
    __shared__ __align__(8) uint64_t s_claim;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    c64_t *park = reinterpret_cast<c64_t *>(smem + kMoveBytes / 2);  // N = 16
    uint32_t tmem = 0;
    if (tid == 0) mbar_init(smem_u32(&s_claim), 1);
    if constexpr (O::kCols > 0) {
        if (warp == 0) tc_alloc(&s_tmem, 2 * O::kCols);
        tc_fence_before();
    }
    __syncthreads();
    if (tid == 0) {
        s_tile[0] = (long long)atomicAdd(work, 1ull);
        mbar_arrive(smem_u32(&s_claim));
    }
    if constexpr (O::kCols > 0) {
        tc_fence_after();
        // this warp's 32 lanes; warps w and w + 4 share them
        tmem = s_tmem + ((uint32_t)(warp & 3) << 21) + (warp >> 2) * O::kCols;
    }
    for (uint32_t n = 0;; ++n) {
        one_wait(smem_u32(&s_claim), n & 1, status, wait_ns);
        const long long g = s_tile[n & 1];
        if (g >= n_tiles) break;
        long long next = 0;
        if (tid == 0) next = (long long)atomicAdd(work, 1ull);
        long long gl = g, sidx = 0;
        const float2 *psi = psi0;
        if (psis) {
            sidx = g / tiles_per_state;
            gl = g - sidx * tiles_per_state;
            psi = reinterpret_cast<const float2 *>(psis[sidx]);
        }
        const uint64_t x0 = x_begin + (uint64_t)gl * O::kShifts;
        c64_t v[32];
        double s;
        if constexpr (O::kShifts > 1) {
            // shift x0 + q in the entries with block bits N - 1 and up equal
            // to q (a last tile past the range repeats its last shift)
            constexpr int kCount = 32 / O::kShifts;
            const uint64_t xl = x_end - 1;
            w32_direct<0, kCount>(v, pair_src(psi, N, x0, 0), tid);
            w32_direct<kCount, kCount>(v, pair_src(psi, N, min(x0 + 1, xl), 0), tid);
            w32_block<O::kBits>(v, smem, tid);
            s = w32_pow(v, alpha);
        } else {
#pragma unroll
            for (int tp = 0; tp < O::kBlocks; ++tp) {
                w32_direct<0, 32, O::kTwice>(v, pair_src(psi, N, x0, tp), tid);
                w32_block<kBlockBits, O::kHalfMove>(v, smem, tid);
                if (tp + 1 < O::kBlocks) {
                    if (tp < O::kTmemBlocks) {
#pragma unroll
                        for (int i = 0; i < 32; i += 4) tmem_put4(tmem + 64 * tp + 2 * i, v + i);
                        tc_wait_st();
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; ++i) park[(i << 8) | tid] = v[i];
                    }
                }
            }
            if constexpr (O::kBlocks == 1) {
                s = w32_pow(v, alpha);
            } else {
                switch (alpha) {
                    case 2: s = one_blocks<N, 2>(v, tmem, park, tid, alpha); break;
                    case 3: s = one_blocks<N, 3>(v, tmem, park, tid, alpha); break;
                    case 4: s = one_blocks<N, 4>(v, tmem, park, tid, alpha); break;
                    default: s = one_blocks<N, O::kTwice ? 0 : -1>(v, tmem, park, tid, alpha);
                }
            }
        }
        s = warp_sum(s);
        if (lane == 0) red[warp] = s;
        __syncthreads();
        // every thread is past its wait for this tile: the next may follow
        if (tid == 0) {
            s_tile[(n + 1) & 1] = *(volatile int *)status != 0 ? n_tiles : next;
            mbar_arrive(smem_u32(&s_claim));
        }
        if (tid < O::kShifts && x0 + (uint64_t)tid < x_end) {
            // N = 13: warp bit 2 is block bit 12, the shift
            constexpr int kWarps = 8 / O::kShifts;
            double t = 0.0;
            for (int w = 0; w < kWarps; ++w) t += red[kWarps * tid + w];
            t *= fp32_scale(O::kTwice ? fp32_doubled(x0 + (uint64_t)tid) : alpha > 4, alpha);
            const uint64_t at = x0 - x_begin + (uint64_t)tid;
            part[(uint64_t)sidx * (x_end - x_begin) + at] = t;
            if (per_x) per_x[at] = t;
        }
    }
    if constexpr (O::kCols > 0) {
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (warp == 0) tc_dealloc(s_tmem, 2 * O::kCols);
    }
}

template <int N>
cudaError_t launch_one_n(const void *psi, const void *const *psis, int nstates, uint64_t xb, uint64_t xe, int alpha,
                         double *part, double *per_x, unsigned long long *work, int *status, long long wait_ns,
                         const DeviceInfo &dev, cudaStream_t st) {
    auto kern = k_one<N>;
    const size_t smem = One<N>::kSmem;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const long long tps = (long long)((xe - xb + One<N>::kShifts - 1) / One<N>::kShifts), n = tps * nstates;
    const int grid = (int)std::min<long long>(n, 2ll * dev.sms);
    kern<<<grid, kBlockThreads, smem, st>>>(reinterpret_cast<const float2 *>(psi), psis, tps, xb, xe, n, alpha, part,
                                            per_x, work, status, wait_ns);
    return cudaGetLastError();
}

}  // namespace

bool one_applies(int N, int elem_bytes) { return elem_bytes == 8 && N >= 13 && N <= 16; }

cudaError_t launch_one(int N, const void *psi, const void *const *psis, int nstates, uint64_t xb, uint64_t xe,
                       int alpha, double *part, double *per_x, unsigned long long *work, int *status,
                       long long wait_ns, const DeviceInfo &dev, cudaStream_t st) {
    switch (N) {
        case 13: return launch_one_n<13>(psi, psis, nstates, xb, xe, alpha, part, per_x, work, status, wait_ns, dev, st);
        case 14: return launch_one_n<14>(psi, psis, nstates, xb, xe, alpha, part, per_x, work, status, wait_ns, dev, st);
        case 15: return launch_one_n<15>(psi, psis, nstates, xb, xe, alpha, part, per_x, work, status, wait_ns, dev, st);
        case 16: return launch_one_n<16>(psi, psis, nstates, xb, xe, alpha, part, per_x, work, status, wait_ns, dev, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace sre
