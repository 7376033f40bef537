// sre_kernels.cu -- CUDA-core XOR-FWHT path of libsre (FP32 and FP64).
//
// Algorithm 1 of the paper: for every shift x, form the XOR-shifted product
// g_x(t) = conj(phi_{t^x}) phi_t, transform it with the unnormalised FWHT over
// t (A_x(z) = <psi|X^x Z^z|psi>, Eq. (Pauli_expect)) and accumulate
// sum_z |A_x(z)|^4; M2 = -log2(S / (d n2^4)) (Eq. (final1), base 2).
//
// Kernels
//   k_convert   element-type conversion of the state (complex128 <-> complex64)
//   k_norm      n2 = <psi|psi> in FP64 + NaN/Inf detection (fixed grid); a
//               single FP32 state with N <= 12 has it from k_small
//   k_small     N <= 12, FP32: one 2^12-entry tile holds 2^(13-N) whole shifts
//               (halved form); the state sits in shared memory; static
//               tile->CTA assignment.  k_small_fx: the same in fixed point
//   k_large     fixed point N >= 15, FP32 N >= 20: persistent two-pass kernel
//               (sre_large.cuh); the sizes between run in sre_mid.cu,
//               sre_one.cu and sre_two.cu
//   k_finalize  fixed-order FP64 sums of the partials, M2 and the status.
// Every reduction has a fixed order, so results are bitwise reproducible and
// do not depend on what else runs on the device.
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "sre_internal.h"
#include "sre_large.cuh"
#include "sre_tile.cuh"
#include "sre_batched.h"
#include "sre_one.h"
#include "sre_two.h"

namespace sre {
using namespace dev;

// ---------------------------------------------------------------- helpers

template <typename Out, typename In>
__global__ void k_convert(const In *__restrict__ src, Out *__restrict__ dst, uint64_t n) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const In v = src[i];
        Out o;
        o.x = (decltype(o.x))v.x;
        o.y = (decltype(o.y))v.y;
        dst[i] = o;
    }
}

// n2 = sum_t |phi_t|^2 (FP64), per-block partials in a fixed grid.
template <typename V>
__global__ void __launch_bounds__(kThreads) k_norm(const V *__restrict__ psi, uint64_t d,
                                                   double *__restrict__ npart,
                                                   int *__restrict__ flags) {
    __shared__ double red[kThreads / 32];
    double s = 0.0;
    int bad = 0;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < d;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const V v = psi[t];
        const double re = (double)v.x, im = (double)v.y;
        if (!isfinite(re) || !isfinite(im)) bad = 1;
        s += re * re + im * im;
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flags, kFlagNonFinite);
    const double b = block_sum(s, red);
    if (threadIdx.x == 0) npart[blockIdx.x] = b;
}

// ------------------------------------------------------------- finalize

// Fixed-order FP64 sum of two segments of partials by one warp: lane l adds
// entries l, l+32, ... of each segment in order, then a fixed shuffle tree.
// Shared by the single-state and the batch finalize, so a state's M2 is
// bitwise the same in either.
__device__ __forceinline__ double warp_sum_segments(const double *p, long long o1, long long n1,
                                                    long long o2, long long n2) {
    const int lane = threadIdx.x & 31;
    double s = 0.0;
    for (long long k = lane; k < n1; k += 32) s += __ldcg(p + o1 + k);
    for (long long k = lane; k < n2; k += 32) s += __ldcg(p + o2 + k);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    return s;  // valid in lane 0
}

__device__ __forceinline__ double m2_from(double S, double n2, int N, bool bad) {
    // M2 = -log2(S / (d n2^4)), in logs so tiny norms do not underflow
    return bad ? __longlong_as_double(0x7ff8000000000000ll)
               : -(log2(S) - (double)N - 4.0 * log2(n2));
}

// Eq. (sre) at integer order alpha: M_alpha = log2(S / (d n2^(2 alpha))) /
// (1 - alpha); order 2 is m2_from.
__device__ __forceinline__ double malpha_from(double S, double n2, int N, int alpha, bool bad) {
    if (alpha == 2) return m2_from(S, n2, N, bad);
    return bad ? __longlong_as_double(0x7ff8000000000000ll)
               : (log2(S) - (double)N - 2.0 * alpha * log2(n2)) / (1.0 - alpha);
}

// One warp: S from the partial segments [o1, o1+n1) and [o2, o2+n2), n2 from
// the norm partials, M2 and the status (by_norm: the entries are FP32, whose n2
// is finite unless an entry is not); host, when given, is pinned memory of
// the caller's that gets the result as well.
__device__ __forceinline__ void finalize_warp(const double *parts, long long o1, long long n1, long long o2,
                                              long long n2c, const double *npart, int nn, int N, int st, bool bad, bool by_norm,
                                              Result *res, Result *host, double *d_m2, int alpha) {
    const double S = warp_sum_segments(parts, o1, n1, o2, n2c);
    const double n2 = warp_sum_segments(npart, 0, nn, 0, 0);
    if ((threadIdx.x & 31) == 0) {
        if (st == 0 && (bad || (by_norm && !isfinite(n2)))) st = SRE_ENONFINITE;
        if (st == 0 && !(n2 > 0.0)) st = SRE_EZERO;
        const double m2 = malpha_from(S, n2, N, alpha, st != 0);
        res->m2 = m2;
        res->S = S;
        res->n2 = n2;
        res->status = st;
        if (host) *host = *res;
        if (d_m2) *d_m2 = m2;
    }
}

__global__ void k_finalize(const double *__restrict__ parts, long long o1, long long n1, long long o2,
                           long long n2c, const double *__restrict__ npart, int nn, int N,
                           const int *flags, const int *status, Result *res, Result *host, double *d_m2,
                           int alpha) {
    finalize_warp(parts, o1, n1, o2, n2c, npart, nn, N, *status, (*flags & kFlagNonFinite) != 0, false, res, host,
                  d_m2, alpha);
}

// What the single-state k_small does besides its tiles: the norm of the state
// that it holds in shared memory (the partials of k_norm, by the same CTAs'
// worth of entries in the same order) and, in the CTA that ends last, the
// finalize.  Two kernels of a few microseconds each, and the gaps before
// them, were most of the device time of a call with N <= 10.
struct SmallTail {
    double *npart = nullptr;  // null: a batch, whose norms and sums are formed elsewhere
    unsigned *ticket = nullptr;
    Result *res = nullptr, *host = nullptr;
    double *d_m2 = nullptr;
};
static_assert(kNormBlocks * kThreads >= kTile, "one entry per thread of k_norm");
// Norm partials with entries; a launch has a CTA for each, however short its
// range: one CTA that forms all sixteen of N = 12 takes 10 us more.
constexpr int small_norm_blocks(int N) { return ((1 << N) + kThreads - 1) / kThreads; }

// ------------------------------------------------------- N <= 12: k_small

// Tile g covers flat indices [g*4096, (g+1)*4096) of the (x - x_begin, t')
// space: x = x_begin + (flat >> NB), t' = flat & (2^NB - 1), NB = N - 1: every
// shift in the halved form, t' being t without the pivot bit (the highest set
// bit of x; x = 0 pairs the two halves of g_0).
template <typename R, int NB>
__global__ void __launch_bounds__(kThreads) k_small(const v2_t<R> *__restrict__ psi,
                                                    const void *const *__restrict__ psis,
                                                    long long tiles_per_state,
                                                    uint64_t x_begin, uint64_t x_end,
                                                    long long ntiles,
                                                    double *__restrict__ part, int alpha, SmallTail tail) {
    // Single state: psis == nullptr.  Several states of the same N: psis[s] is
    // state s and tiles are numbered state-major.  Tile g's sum goes to
    // part[g] (fixed-order tree inside the tile), so a state's partials do not
    // depend on the grid or on the other states of a batch.
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using V = v2_t<R>;
    V *psi_s = reinterpret_cast<V *>(smem_raw);
    V *bufA = psi_s + kTileSlots;
    V *bufB = bufA + kTileSlots;
    __shared__ double red[kThreads / 32];
    constexpr int N = NB + 1;
    constexpr int d = 1 << N;
    const int tid = threadIdx.x;

    long long cur = -1;
    for (long long g = blockIdx.x; g < ntiles; g += gridDim.x) {
        const long long sidx = psis ? g / tiles_per_state : 0;
        const long long gl = g - sidx * tiles_per_state;
        if (sidx != cur) {
            const V *src = psis ? reinterpret_cast<const V *>(psis[sidx]) : psi;
            __syncthreads();
            for (int t = tid; t < d; t += kThreads) psi_s[pad(t)] = src[t];
            __syncthreads();
            cur = sidx;
        }
        cx_t<R> v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const uint64_t flat = ((uint64_t)gl << kTileBits) | (uint64_t)elem<0>(tid, i);
            const uint64_t x = x_begin + (flat >> NB);
            if (x < x_end) {
                const int xe = x ? (int)x : d >> 1;
                const int lo = (int)(flat & ((1u << NB) - 1)) & ((1 << (31 - __clz(xe))) - 1);
                const int t = (((int)(flat & ((1u << NB) - 1)) - lo) << 1) | lo;
                v[i] = x ? pair_value<R, false>(psi_s[pad(t ^ xe)], psi_s[pad(t)])
                         : pair_value<R, true>(psi_s[pad(t ^ xe)], psi_s[pad(t)]);
                v[i] = Cx<R>::add(v[i], v[i]);  // fp32_doubled
            } else {
                v[i] = Cx<R>::zero();
            }
        }
        tile_fwht<NB, R>(v, bufA, bufB, tid);
        // block_sum's barriers also protect bufB before the next tile
        const double s = block_sum((double)sum_order<R>(v, alpha), red);
        if (tid == 0) part[g] = s;
    }
    if (!tail.npart) return;
    constexpr int kUsed = small_norm_blocks(N);
    for (int b = blockIdx.x; b < kUsed; b += gridDim.x) {
        const int t = b * kThreads + tid;
        // a CTA without a tile has no copy of the state
        const V e = t >= d ? V{0, 0} : cur < 0 ? psi[t] : psi_s[pad(t)];
        const double re = (double)e.x, im = (double)e.y;
        __syncthreads();  // red is free
        const double s = block_sum(re * re + im * im, red);
        if (tid == 0) tail.npart[b] = s;
    }
    __shared__ bool last;
    if (tid == 0) {
        __threadfence();
        last = atomicAdd(tail.ticket, 1u) + 1u == gridDim.x;
        __threadfence();
    }
    __syncthreads();
    if (last && tid < 32)
        finalize_warp(part, 0, ntiles, 0, 0, tail.npart, kUsed, N, 0, false, true, tail.res, tail.host, tail.d_m2,
                      alpha);
}

// The same in the fixed-point mode: factors straight from global memory (the
// state stays in L1), bits 8-11 first, one move buffer, so that two CTAs fit
// an SM.
template <int NB>
__global__ void __launch_bounds__(kThreads, 2) k_small_fx(const double2 *__restrict__ psi0,
                                                          const void *const *__restrict__ psis,
                                                          long long tiles_per_state, uint64_t x_begin, uint64_t x_end,
                                                          long long ntiles, double *__restrict__ part, int alpha) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2 *buf = reinterpret_cast<double2 *>(smem_raw);
    __shared__ double red[kThreads / 32];
    __shared__ FxShared sh;
    constexpr int d = 2 << NB;
    const int tid = threadIdx.x;
    for (long long g = blockIdx.x; g < ntiles; g += gridDim.x) {
        const long long sidx = psis ? g / tiles_per_state : 0;
        const long long gl = g - sidx * tiles_per_state;
        const double2 *psi = psis ? reinterpret_cast<const double2 *>(psis[sidx]) : psi0;
        cx_t<fx> v[16];
        auto value = [&](int i, auto with_zero) {
            const uint64_t flat = ((uint64_t)gl << kTileBits) | (uint64_t)elem<2>(tid, i);
            const uint64_t x = x_begin + (flat >> NB);
            if (x >= x_end) return Cx<fx>::zero();
            const int xe = x ? (int)x : d >> 1, tt = (int)(flat & ((1u << NB) - 1));
            const int lo = tt & ((1 << (31 - __clz(xe))) - 1), t = ((tt - lo) << 1) | lo;
            const double2 b = __ldg(psi + (t ^ xe)), a = __ldg(psi + t);
            if constexpr (decltype(with_zero)::value)
                if (!x) return pair_value<fx, true>(b, a);
            return pair_value<fx, false>(b, a);
        };
        // the first tile alone holds x = 0
        if (gl == 0 && x_begin == 0) {
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = value(i, std::true_type());
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = value(i, std::false_type());
        }
        const FxExp u = fx_tile<NB>(v, buf, tid, sh);
        const double s = block_sum(sum_order<fx>(v, alpha), red);
        if (tid == 0) part[g] = fx_scale(s, alpha, u.c);
    }
}

// M_alpha from a reduced sum and a norm (sums of shards added elsewhere).
__global__ void k_malpha_from_sums(const double *S, const double *n2, int N, int alpha, double *out) {
    const double s = *S, n = *n2;
    const bool bad = !(s > 0.0) || !(n > 0.0) || !isfinite(s) || !isfinite(n);
    *out = malpha_from(s, n, N, alpha, bad);
}

__global__ void k_copy_sums(const Result *res, double *out2) {
    out2[0] = res->S;
    out2[1] = res->n2;
}

// ------------------------------------------------------------ host side

cudaError_t query_device(DeviceInfo *info) {
    cudaError_t e = cudaGetDevice(&info->device);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&info->sms, cudaDevAttrMultiProcessorCount, info->device);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&info->l2_bytes, cudaDevAttrL2CacheSize, info->device);
    if (e != cudaSuccess) return e;
    return cudaDeviceGetAttribute(&info->max_smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin,
                                  info->device);
}

// deterministic pseudo-random amplitudes for timing runs (values irrelevant)
template <typename V>
__global__ void k_fill_synthetic(V *p, uint64_t n) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t h = (i + 1) * 0x9E3779B97F4A7C15ull;
        h ^= h >> 31;
        h *= 0xBF58476D1CE4E5B9ull;
        h ^= h >> 29;
        V v;
        v.x = (decltype(v.x))((double)(h & 0xFFFFFF) / 16777216.0 - 0.5);
        v.y = (decltype(v.y))((double)((h >> 24) & 0xFFFFFF) / 16777216.0 - 0.5);
        p[i] = v;
    }
}

cudaError_t enqueue_fill_synthetic(void *buf, int N, sre_dtype_t dtype, cudaStream_t st) {
    const uint64_t d = 1ull << N;
    const int grid = (int)std::min<uint64_t>((d + 255) / 256, 4096);
    if (dtype == SRE_C128)
        k_fill_synthetic<double2><<<grid, 256, 0, st>>>(reinterpret_cast<double2 *>(buf), d);
    else
        k_fill_synthetic<float2><<<grid, 256, 0, st>>>(reinterpret_cast<float2 *>(buf), d);
    return cudaGetLastError();
}

bool large_cfg_fits(const Workspace &ws, const LargeCfg &c, int N) {
    if (c.C_log < 0 || c.C_log > 3 || c.R < 2 || c.R > kMaxRing || c.D < 1 || c.D >= c.R) return false;
    const int h2 = N - kTileBits - 1;
    if (c.G2_log < 0 || c.G2_log > h2 || c.B1_log < 0 || c.B1_log > h2) return false;
    const size_t ring = (size_t)c.R * ((size_t)1 << c.C_log) * ((size_t)ws.elem_bytes << (N - 1));
    const size_t P2 = ((size_t)1 << c.C_log) << (h2 - c.G2_log);
    return ring <= ws.scratch_bytes && (size_t)c.R * P2 * 8 <= ws.item_part_cap;
}

// Ring / chunk configuration for the two-pass kernel.  About grid / P1
// chunks are in pass 1 at any time (P1 = 2^h2 items per chunk), so pass 2
// lags D = that + 1 chunks behind and the ring holds R = 2 D + 1 chunks:
// pass-2 items then find their chunk finished and pass-1 items find their
// slot free.  The chunk size C (shifts sharing one pass-1 partner block) is
// the largest power of two up to 8 whose ring R * C * elem * 2^(N - 1)
// stays within 60% of L2, so the inter-pass traffic stays on chip.
LargeCfg choose_large_cfg(const DeviceInfo &dev, int N, int elem_bytes) {
    LargeCfg c;
    const int h2 = N - kTileBits - 1;
    const double per_x = (double)elem_bytes * (double)(1ull << (N - 1));
    const double budget = std::max(24.0 * (1 << 20), 0.6 * (double)dev.l2_bytes);
    c.grid = std::max(1, dev.sms * 2);
    const int P1 = 1 << h2;
    const int inflight = (c.grid + P1 - 1) / P1;
    c.D = std::min(inflight + 1, kMaxRing / 2 - 1);
    c.R = 2 * c.D + 1;
    int C_log = 3;
    while (C_log > 0 && (double)c.R * (double)(1 << C_log) * per_x > budget) --C_log;
    c.C_log = C_log;
    c.G2_log = std::min(C_log, h2);
    c.stage1 = 1;
    c.stage2 = 1;
    // items of four tiles or more: tiles by tensor copy (FP32, h2 = 7 and 8, and
    // the tensor-core kernel) overlap the copy of tile g + 2 with tile g
    if (elem_bytes == 8 && h2 >= 5 && h2 <= 8) c.G2_log = std::min(C_log + 2, h2);
    c.B1_log = 0;
    return c;
}

// The tensor-core kernel's ring: eight shifts per chunk, so that one pass-1
// operand build serves eight, and as many slots as the tuning scratch (192 MB)
// holds, with pass 2 a third of the ring behind.  One CTA per SM holds a
// pass-1 item for far longer than the L2-sized rings of choose_large_cfg last,
// and pass 1 then waits for slots.  fp16_split, 2^31 to 2^33 halved entries,
// L2-sized ring -> this one: N = 16 5.68 -> 4.75 ms, 17 12.9 -> 7.5, 18 19.7 -> 12.9,
// 19 18.6 -> 12.7, 20 18.4 -> 13.1.  Six slots at least: a workspace with less
// scratch takes fewer shifts per chunk, and below that the general rule.
static LargeCfg choose_tc_cfg(const DeviceInfo &dev, const Workspace &ws, int N) {
    LargeCfg c = choose_large_cfg(dev, N, 8);
    const size_t ring = std::min(ws.scratch_bytes, kTuneScratch);
    for (int C_log = 3; C_log >= 0; --C_log) {
        const int R = (int)std::min<size_t>(kMaxRing - 1, ring / ((size_t)8 << (N - 1 + C_log)));
        if (R < 6) continue;
        c.C_log = C_log;
        c.R = R;
        c.D = R / 3;
        c.G2_log = std::min(5, N - 1 - kTileBits);
        break;
    }
    return c;
}

// FP32 at N = 20: one shift per chunk, block pairs and tiles by bulk and tensor
// copies, eight blocks and eight tiles per item, and all the slots that the
// tuning scratch holds (47 of 4 MB).  1.90 s for a whole state, against 1.98 s
// by the item-list kernel of sre_two.cu.  A short ring makes it wait: a server's
// slots (96 MB) take 2.46 s, 8192 shifts 19.1 ms in place of 14.9 (the item-list
// kernel with that ring 2.36 s and 22.2 ms).  Below 23 slots the general rule.
// Fewer than 16 shifts take smaller items, or most SMs have none (one shift 56
// against 68 us, 16 shifts 90 in either).
constexpr int kFp32LargeN = 20, kFp32Ring = 47;
static LargeCfg choose_fp32_20_cfg(const DeviceInfo &dev, const Workspace &ws, uint64_t shifts) {
    LargeCfg c = choose_large_cfg(dev, kFp32LargeN, 8);
    const int R = (int)std::min<size_t>(kFp32Ring, ws.scratch_bytes / ((size_t)8 << (kFp32LargeN - 1)));
    if (R >= 23) {
        c.C_log = 0;
        c.R = R;
        c.D = (R - 1) / 2;
        c.G2_log = shifts < 16 ? 2 : 3;
        c.B1_log = shifts < 16 ? 0 : 3;
    }
    return c;
}

LargeCfg choose_main_cfg(const DeviceInfo &dev, const Workspace &ws, int N, sre_mode_t mode, uint64_t shifts) {
    const int eb = mode == SRE_MODE_FP64 ? 16 : 8;
    if (mode == SRE_MODE_FP32 && N == kFp32LargeN) return choose_fp32_20_cfg(dev, ws, shifts);
    // fewer than 64 shifts leave most SMs without an item of the large chunks:
    // one shift of N = 18 takes 87 us in small ones, 108 in large ones; 48 shifts
    // 105 and 121, 128 shifts 154 and 144
    if (tc_mode_available(mode) && tc_applies(N, 2, nullptr) && shifts >= 64) return choose_tc_cfg(dev, ws, N);
    return choose_large_cfg(dev, N, eb);
}

LargeCfg tuning_base_cfg(const DeviceInfo &dev, const Workspace &ws, int N, sre_mode_t mode, const sre_tuning_t &t,
                         uint64_t shifts) {
    if (t.x_batch_log >= 0 || t.ring_slots >= 0 || t.lag >= 0)
        return choose_large_cfg(dev, N, mode == SRE_MODE_FP64 ? 16 : 8);
    return choose_main_cfg(dev, ws, N, mode, shifts);
}

// FP32 shifts by sre_two.cu: at N = 20 only beside the tensor-core kernel.
static bool takes_two(int N, int elem_bytes, int tc_kind) {
    return two_applies(N, elem_bytes) && (N < kFp32LargeN || tc_kind);
}

void workspace_free(Workspace *ws) {
    if (ws->ev_begin) cudaEventDestroy(ws->ev_begin);
    if (ws->ev_end) cudaEventDestroy(ws->ev_end);
    cudaFree(ws->npart);
    cudaFree(ws->part);
    cudaFree(ws->scratch);
    cudaFree(ws->item_part);
    cudaFree(ws->chunk_sum);
    cudaFree(ws->counters);
    cudaFree(ws->work);
    cudaFree(ws->result);
    cudaFree(ws->conv);
    cudaFree(ws->tc_e);
    cudaFree(ws->tc_bn);
    cudaFree(ws->fx_exp);
    *ws = Workspace();
}

cudaError_t workspace_alloc(Workspace *ws, const DeviceInfo &dev, int N_max, int elem_bytes,
                            sre_mode_t mode, size_t scratch_floor) {
    (void)mode;
    *ws = Workspace();
    ws->N_max = N_max;
    ws->elem_bytes = elem_bytes;
    cudaError_t e;
#define SRE_TRY(x)                  \
    do {                            \
        e = (x);                    \
        if (e != cudaSuccess) {     \
            workspace_free(ws);     \
            return e;               \
        }                           \
    } while (0)
    SRE_TRY(cudaMalloc(&ws->npart, sizeof(double) * kNormBlocks));
    ws->part_cap = kTile;  // one partial per tile of an N <= 12 state
    SRE_TRY(cudaMalloc(&ws->part, sizeof(double) * ws->part_cap));
    SRE_TRY(cudaMalloc(&ws->work, kWorkBytes + kFlagBytes));
    ws->flags = reinterpret_cast<int *>(ws->work + kWorkBytes / 8);
    ws->status = ws->flags + 1;
    SRE_TRY(cudaMalloc(&ws->result, sizeof(Result)));
    if (N_max > kTileBits) {
        // sizes for every N up to N_max, and with the ring of one qubit more
        // room for tuned configurations: chunks of a single shift, up to
        // kMaxRing ring slots, a scratch ring of at least scratch_floor bytes
        size_t scratch = scratch_floor, item_cap = 0;
        const size_t chunk_cap = ((size_t)1 << N_max) + 4;
        for (int n = kTileBits + 1; n <= N_max + 1; ++n) {
            const LargeCfg c = choose_large_cfg(dev, n, elem_bytes);
            scratch = std::max(scratch, (size_t)c.R * ((size_t)1 << c.C_log) * ((size_t)elem_bytes << (n - 1)));
            // R * P2 per-warp partials (8 warps, P2 <= 8 * 2^h2)
            item_cap = std::max(item_cap, (size_t)std::max(c.R, kMaxRing) * ((size_t)8 << (n - kTileBits - 1)) * 8);
        }
        ws->scratch_bytes = scratch;
        ws->item_part_cap = item_cap;
        ws->chunk_cap = chunk_cap;
        SRE_TRY(cudaMalloc(&ws->scratch, scratch));
        SRE_TRY(cudaMalloc(&ws->item_part, sizeof(double) * item_cap));
        SRE_TRY(cudaMalloc(&ws->chunk_sum, sizeof(double) * chunk_cap));
        SRE_TRY(cudaMalloc(&ws->counters, sizeof(unsigned) * 3 * chunk_cap));
        ws->tc_cap = 1 << (N_max - kTileBits);
        SRE_TRY(cudaMalloc(&ws->tc_e, sizeof(int) * ws->tc_cap));
        SRE_TRY(cudaMalloc(&ws->tc_bn, sizeof(double) * ws->tc_cap));
        if (elem_bytes == 16) {
            // unit and bound of every block in the ring: R * C * 2^h2 of each
            ws->fx_cap = item_cap / 8;
            SRE_TRY(cudaMalloc(&ws->fx_exp, sizeof(short) * 2 * ws->fx_cap));
        }
    }
#undef SRE_TRY
    return cudaSuccess;
}

template <typename R, int NB>
static cudaError_t launch_small_nb(const void *psi, const void *const *psis, int nstates,
                                   uint64_t x_begin, uint64_t x_end, double *part, int part_cap,
                                   const DeviceInfo &dev, cudaStream_t st, int *nparts,
                                   int forced_grid, int alpha, const SmallTail &tail) {
    constexpr bool kFx = sizeof(cx_t<R>) == 16;
    const size_t smem = (size_t)(kFx ? 1 : 3) * kTileSlots * sizeof(v2_t<R>);
    cudaError_t e;
    if constexpr (kFx)
        e = cudaFuncSetAttribute(k_small_fx<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    else
        e = cudaFuncSetAttribute(k_small<R, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const uint64_t flat = (x_end - x_begin) << NB;
    const long long tps = (long long)((flat + kTile - 1) >> kTileBits);
    const long long ntiles = tps * nstates;
    if (ntiles > part_cap) return cudaErrorInvalidValue;
    int grid = forced_grid > 0 ? forced_grid : (int)std::min<long long>(ntiles, (long long)dev.sms * 2);
    if (grid < 1) return cudaErrorInvalidValue;
    if (tail.npart) grid = std::max(grid, small_norm_blocks(NB + 1));
    if constexpr (kFx)
        k_small_fx<NB><<<grid, kThreads, smem, st>>>(reinterpret_cast<const double2 *>(psi), psis, tps, x_begin, x_end,
                                                     ntiles, part, alpha);
    else
        k_small<R, NB><<<grid, kThreads, smem, st>>>(reinterpret_cast<const float2 *>(psi), psis, tps, x_begin, x_end,
                                                     ntiles, part, alpha, tail);
    *nparts = (int)ntiles;
    return cudaGetLastError();
}

template <typename R>
static cudaError_t launch_small(int N, const void *psi, const void *const *psis, int nstates,
                                uint64_t xb, uint64_t xe, double *part, int part_cap,
                                const DeviceInfo &dev, cudaStream_t st, int *nparts,
                                int forced_grid, int alpha, const SmallTail &tail = SmallTail()) {
    switch (N) {
#define SRE_CASE(n) \
    case n: return launch_small_nb<R, n - 1>(psi, psis, nstates, xb, xe, part, part_cap, dev, st, nparts, forced_grid, alpha, tail);
        SRE_CASE(1) SRE_CASE(2) SRE_CASE(3) SRE_CASE(4) SRE_CASE(5) SRE_CASE(6)
        SRE_CASE(7) SRE_CASE(8) SRE_CASE(9) SRE_CASE(10) SRE_CASE(11) SRE_CASE(12)
#undef SRE_CASE
        default: return cudaErrorInvalidValue;
    }
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link
// dependency on the driver library).
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }();
    return fn;
}

// The scratch ring of a launch as a 2-D FP32 array: 8192 columns (the 4096
// complex entries of one block t'_h) by R * C * 2^h2 rows, 32 KB apart; boxes
// of 32 FP32 columns (128 bytes, the swizzle span) by 2^h2 rows.
cudaError_t encode_p2_tmap(LargeArgs &a) {
    auto enc = tensor_map_encoder();
    if (!enc) return cudaErrorNotSupported;
    if (a.h2 < 7 || a.h2 > 8 || ((uintptr_t)a.scratch & 15)) return cudaErrorInvalidValue;
    const cuuint64_t rows = (cuuint64_t)a.R << (a.C_log + a.h2);
    if (rows > 0xFFFFFFFFull) return cudaErrorInvalidValue;
    const cuuint64_t dims[2] = {2ull * kTile, rows};
    const cuuint64_t strides[1] = {(cuuint64_t)kTile * sizeof(float2)};
    const cuuint32_t box[2] = {32u, 1u << a.h2};
    const cuuint32_t estr[2] = {1u, 1u};
    const CUresult r = enc(&a.tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, a.scratch, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <typename R, int H2>
static cudaError_t launch_large_h(const LargeArgs &a, int grid, cudaStream_t st) {
    const size_t smem = large_smem_bytes<R, H2>();
    auto kern = k_large<R, H2>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if constexpr (large_uses_tma<R, H2>()) {
        LargeArgs b = a;
        if ((e = encode_p2_tmap(b)) != cudaSuccess) return e;
        kern<<<grid, kThreads, smem, st>>>(b);
    } else {
        kern<<<grid, kThreads, smem, st>>>(a);
    }
    return cudaGetLastError();
}

// FP32: N >= 20 (smaller sizes run in sre_one.cu and sre_two.cu); fixed point:
// N >= 15.
template <typename R>
static cudaError_t launch_large(const LargeArgs &a, int grid, cudaStream_t st) {
    switch (a.h2) {
#define SRE_CASE(n) \
    case n: return launch_large_h<R, n>(a, grid, st);
        SRE_CASE(7) SRE_CASE(8) SRE_CASE(9) SRE_CASE(10) SRE_CASE(11)
#undef SRE_CASE
#define SRE_CASE(n) \
    case n: if constexpr (sizeof(cx_t<R>) == 16) return launch_large_h<R, n>(a, grid, st); break;
        SRE_CASE(2) SRE_CASE(3) SRE_CASE(4) SRE_CASE(5) SRE_CASE(6)
#undef SRE_CASE
    }
    return cudaErrorInvalidValue;
}

// Fill LargeArgs for the shift range [xb, xe).
static cudaError_t make_large_args(LargeArgs *a, const Workspace &ws, const DeviceInfo &dev,
                                   const void *psi, int N, uint64_t xb, uint64_t xe,
                                   int elem_bytes, size_t chunk_off, double *per_x,
                                   long long wait_ns, const LargeCfg &c, int *grid) {
    LargeArgs &A = *a;
    A.psi = psi;
    A.psis = nullptr;
    A.chunks_per_state = 0;
    A.fx_exp = ws.fx_exp;
    A.fx_cap = ws.fx_cap;
    A.tc_e = ws.tc_e;
    A.N = N;
    A.h2 = N - kTileBits - 1;
    A.x_begin = xb;
    A.x_end = xe;
    A.C_log = c.C_log;
    A.R = c.R;
    A.G2_log = std::min(c.G2_log, A.h2);
    A.x0 = xb & ~((1ull << c.C_log) - 1);
    A.n_chunks = (long long)((xe - A.x0 + (1ull << c.C_log) - 1) >> c.C_log);
    A.D = (int)std::max<long long>(1, std::min<long long>(std::min(c.D, c.R - 1), A.n_chunks));
    if (A.R < 2) return cudaErrorInvalidValue;
    A.B1_log = std::max(0, std::min(c.B1_log, A.h2));
    A.stage1 = c.stage1;
    A.stage2 = c.stage2;
    A.alpha = 2;
    A.P1 = 1 << (A.h2 - A.B1_log);
    A.P2 = (1 << c.C_log) << (A.h2 - A.G2_log);
    A.n_items = A.n_chunks * (long long)(A.P1 + A.P2);
    const size_t need_scratch = (size_t)c.R * ((size_t)1 << c.C_log) * ((size_t)elem_bytes << (N - 1));
    if (need_scratch > ws.scratch_bytes || chunk_off + (size_t)A.n_chunks > ws.chunk_cap ||
        (size_t)c.R * A.P2 * 8 > ws.item_part_cap ||
        (elem_bytes == 16 && (size_t)c.R << (c.C_log + A.h2) > ws.fx_cap))
        return cudaErrorInvalidValue;
    A.scratch = ws.scratch;
    A.item_part = ws.item_part;
    A.chunk_sum = ws.chunk_sum + chunk_off;
    A.done1 = ws.counters + chunk_off;
    A.done2 = ws.counters + ws.chunk_cap + chunk_off;
    A.freed = ws.counters + 2 * ws.chunk_cap + chunk_off;
    A.work = ws.work + 1;
    A.per_x = per_x;
    A.status = ws.status;
    A.wait_ns = wait_ns;
    *grid = (int)std::max<long long>(1, std::min<long long>(c.grid, A.n_items));
    return cudaSuccess;
}

cudaError_t enqueue_copy_sums(const Workspace &ws, double *d_out2, cudaStream_t stream) {
    k_copy_sums<<<1, 1, 0, stream>>>(ws.result, d_out2);
    return cudaGetLastError();
}

// The workspace's words that start from zero: flags, status and ticket, which
// follow the work-queue counters (with_work) in one allocation.
static cudaError_t clear_words(const Workspace &ws, bool with_work, cudaStream_t st) {
    return with_work ? cudaMemsetAsync(ws.work, 0, kWorkBytes + kFlagBytes, st)
                     : cudaMemsetAsync(ws.flags, 0, kFlagBytes, st);
}

// One FP32 state with N <= 12, shifts [xb, xe): one kernel, result and all.
static cudaError_t enqueue_small(const Workspace &ws, const DeviceInfo &dev, const void *psi, int N, uint64_t xb,
                                 uint64_t xe, cudaStream_t st, double *d_m2, int alpha) {
    const cudaError_t e = clear_words(ws, false, st);
    if (e != cudaSuccess) return e;
    SmallTail tail;
    tail.npart = ws.npart;
    tail.ticket = reinterpret_cast<unsigned *>(ws.flags) + 2;
    tail.res = ws.result;
    tail.host = ws.host_result;
    tail.d_m2 = d_m2;
    int np = 0;
    return launch_small<float>(N, psi, nullptr, 1, xb, xe, ws.part, ws.part_cap, dev, st, &np, 0, alpha, tail);
}

template <typename R>
static cudaError_t enqueue_m2_t(const Workspace &ws, const DeviceInfo &dev, const void *psi, int N,
                                uint64_t x_begin, uint64_t x_end, cudaStream_t st, double *d_m2,
                                double *d_per_x, long long wait_ns, LargeCfg *cfg_override,
                                int tc_kind, int alpha) {
    cudaError_t e;
    constexpr bool kFx = sizeof(cx_t<R>) == 16;
    const uint64_t d = 1ull << N;
    if constexpr (!kFx)
        if (N <= kTileBits) {
            if (ws.ev_begin && (e = cudaEventRecord(ws.ev_begin, st)) != cudaSuccess) return e;
            if ((e = enqueue_small(ws, dev, psi, N, x_begin, x_end, st, d_m2, alpha)) != cudaSuccess) return e;
            if (ws.ev_end && (e = cudaEventRecord(ws.ev_end, st)) != cudaSuccess) return e;
            ws.main_kernel = "k_small";
            ws.launches += 1;
            return cudaSuccess;
        }
    if ((e = clear_words(ws, N > kTileBits, st)) != cudaSuccess) return e;
    k_norm<<<kNormBlocks, kThreads, 0, st>>>(reinterpret_cast<const v2_t<R> *>(psi), d, ws.npart, ws.flags);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    ws.launches += 2;  // k_norm + k_finalize
    const double *parts = nullptr;
    long long nparts = 0, seg1 = 0;  // [0, seg1) shifts below 4096 beside the tensor-core kernel's [seg1, nparts)
    if (N <= kTileBits) {
        int np = 0;
        if (ws.ev_begin && (e = cudaEventRecord(ws.ev_begin, st)) != cudaSuccess) return e;
        if ((e = launch_small<R>(N, psi, nullptr, 1, x_begin, x_end, ws.part, ws.part_cap, dev, st,
                                 &np, 0, alpha)) != cudaSuccess)
            return e;
        if (ws.ev_end && (e = cudaEventRecord(ws.ev_end, st)) != cudaSuccess) return e;
        ws.main_kernel = "k_small";
        ws.launches += 1;
        parts = ws.part;
        nparts = np;
    } else {
        const int eb = (int)sizeof(v2_t<R>);
        // every shift in one launch, or with the tensor-core kernel on the
        // shifts from 4096 up those below it
        const bool tc = tc_kind && tc_applies(N, alpha, psi);
        const uint64_t split = tc ? std::min<uint64_t>(std::max<uint64_t>(x_begin, kTile), x_end) : x_end;
        const bool single_pass = one_applies(N, eb) || mid_applies(N, eb);
        const sre_mode_t mode = kFx ? SRE_MODE_FP64 : tc_kind ? SRE_MODE_FP16_SPLIT : SRE_MODE_FP32;
        const LargeCfg main = cfg_override ? *cfg_override : choose_main_cfg(dev, ws, N, mode, x_end - split + (tc ? 0 : split - x_begin));
        // chunk counters: not for a shift per CTA
        if ((tc || !single_pass) &&
            (e = cudaMemsetAsync(ws.counters, 0, sizeof(unsigned) * 3 * ws.chunk_cap, st)) != cudaSuccess)
            return e;
        size_t chunks = 0;
        if (x_begin < split) {
            const bool timed = split == x_end;
            if (timed && ws.ev_begin && (e = cudaEventRecord(ws.ev_begin, st)) != cudaSuccess) return e;
            const char *name;
            if (single_pass) {
                // a shift in one CTA, one partial per shift
                name = kFx ? "k_mid" : "k_one";
                chunks = (size_t)(split - x_begin);
                if (chunks > ws.chunk_cap) return cudaErrorInvalidValue;
                if constexpr (kFx)
                    e = launch_mid(N, psi, nullptr, 1, (long long)chunks, x_begin, alpha, ws.chunk_sum, d_per_x, dev, st);
                else
                    e = launch_one(N, psi, nullptr, 1, x_begin, split, alpha, ws.chunk_sum, d_per_x, ws.work + 2,
                                   ws.status, wait_ns, dev, st);
            } else if (takes_two(N, eb, tc_kind)) {
                name = "k_two";
                const LargeCfg c = choose_two_cfg(dev, ws, N);
                e = launch_two(ws, c, N, psi, nullptr, 1, x_begin, split, alpha, ws.chunk_sum, ws.counters,
                               ws.chunk_cap, ws.chunk_cap, ws.work + 2, d_per_x, wait_ns, st);
                chunks = (size_t)two_layout(ws, c, N, x_begin, split).n_chunks;
            } else {
                name = "k_large";
                LargeArgs a;
                int grid = 0;
                if ((e = make_large_args(&a, ws, dev, psi, N, x_begin, split, eb, 0, d_per_x, wait_ns,
                                         main, &grid)) != cudaSuccess)
                    return e;
                a.alpha = alpha;
                e = launch_large<R>(a, grid, st);
                chunks = (size_t)a.n_chunks;
            }
            if (e != cudaSuccess) return e;
            if (timed && ws.ev_end && (e = cudaEventRecord(ws.ev_end, st)) != cudaSuccess) return e;
            if (timed) ws.main_kernel = name;
            ws.launches += 1;
            if (tc) seg1 = (long long)chunks;
        }
        if (tc && split < x_end) {
            LargeArgs a;
            int grid = 0;
            if ((e = make_large_args(&a, ws, dev, psi, N, split, x_end, eb, chunks,
                                     d_per_x ? d_per_x + (split - x_begin) : nullptr, wait_ns, main,
                                     &grid)) != cudaSuccess)
                return e;
            a.alpha = alpha;
            if ((e = launch_large_tc(a, ws, dev, grid, st, tc_kind)) != cudaSuccess) return e;
            ws.launches += 1;
            chunks += (size_t)a.n_chunks;
        }
        parts = ws.chunk_sum;
        nparts = (long long)chunks;
    }
    k_finalize<<<1, 32, 0, st>>>(parts, 0, seg1, seg1, nparts - seg1, ws.npart, kNormBlocks, N,
                                 ws.flags, ws.status, ws.result, ws.host_result, d_m2, alpha);
    return cudaGetLastError();
}

// M2 of one complex64 state in FP32 for N <= 16 (no allocation): the
// single-state path's kernels, on scratch that the caller hands in.
cudaError_t enqueue_m2_fixed(const Workspace &ws, const DeviceInfo &dev, const void *psi, int N, cudaStream_t st,
                             double *d_m2, long long wait_ns) {
    cudaError_t e;
    const uint64_t d = 1ull << N;
    if (N <= kTileBits) return enqueue_small(ws, dev, psi, N, 0, d, st, d_m2, 2);
    if (!one_applies(N, 8) || d > ws.chunk_cap) return cudaErrorInvalidValue;
    if ((e = clear_words(ws, true, st)) != cudaSuccess) return e;
    k_norm<<<kNormBlocks, kThreads, 0, st>>>(reinterpret_cast<const float2 *>(psi), d, ws.npart, ws.flags);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = launch_one(N, psi, nullptr, 1, 0, d, 2, ws.chunk_sum, nullptr, ws.work + 2, ws.status, wait_ns, dev,
                        st)) != cudaSuccess)
        return e;
    k_finalize<<<1, 32, 0, st>>>(ws.chunk_sum, 0, (long long)d, (long long)d, 0, ws.npart, kNormBlocks, N, ws.flags,
                                 ws.status, ws.result, nullptr, d_m2, 2);
    return cudaGetLastError();
}

cudaError_t enqueue_m2(const Workspace &ws, const DeviceInfo &dev, const void *d_state,
                       sre_dtype_t dtype, int N, uint64_t x_begin, uint64_t x_end,
                       sre_mode_t mode, cudaStream_t stream, double *d_m2, double *d_per_x,
                       long long wait_ns, LargeCfg *cfg_override, int alpha) {
    const bool fp64 = (mode == SRE_MODE_FP64);
    const int want = fp64 ? SRE_C128 : SRE_C64;
    const void *psi = d_state;
    const uint64_t d = 1ull << N;
    if ((int)dtype != want) {
        const size_t need = (size_t)d * (fp64 ? 16 : 8);
        if (!ws.conv || ws.conv_bytes < need) return cudaErrorInvalidValue;
        const int grid = (int)std::min<uint64_t>((d + kThreads - 1) / kThreads, 4096);
        if (fp64)
            k_convert<double2, float2><<<grid, kThreads, 0, stream>>>(
                reinterpret_cast<const float2 *>(d_state), reinterpret_cast<double2 *>(ws.conv), d);
        else
            k_convert<float2, double2><<<grid, kThreads, 0, stream>>>(
                reinterpret_cast<const double2 *>(d_state), reinterpret_cast<float2 *>(ws.conv), d);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        ws.launches += 1;
        psi = ws.conv;
    }
    const int tc_kind = mode == SRE_MODE_BF16_SPLIT ? 1 : mode == SRE_MODE_FP16_SPLIT ? 2 : 0;
    if (fp64)
        return enqueue_m2_t<fx>(ws, dev, psi, N, x_begin, x_end, stream, d_m2, d_per_x, wait_ns,
                                    cfg_override, 0, alpha);
    return enqueue_m2_t<float>(ws, dev, psi, N, x_begin, x_end, stream, d_m2, d_per_x, wait_ns,
                               cfg_override, tc_kind, alpha);
}

// --------------------------------------------------------- wait self test

// One thread waits on a counter nothing increments; records the outcome.
__global__ void k_wait_selftest(const unsigned *counter, int *status, long long wait_ns) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        if (wait_counter(counter, 1u, status, wait_ns)) atomicCAS(status, 0, -1);
    }
}

cudaError_t run_wait_selftest(long long wait_ns, cudaStream_t st, int *status_out) {
    unsigned *counter = nullptr;
    int *status = nullptr;
    cudaError_t e = cudaMalloc(&counter, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMalloc(&status, sizeof(int));
    if (e == cudaSuccess) e = cudaMemsetAsync(counter, 0, sizeof(unsigned), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(status, 0, sizeof(int), st);
    if (e == cudaSuccess) {
        k_wait_selftest<<<1, 32, 0, st>>>(counter, status, wait_ns);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(status_out, status, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(counter);
    cudaFree(status);
    return e;
}

// ------------------------------------------------------------------ batch

// n2 of several states (state s = blockIdx.y, its size from Ns[s]);
// partials in npart[s * kNormBlocks + b], flags[s] |= non-finite.
template <typename R>
__global__ void __launch_bounds__(kThreads) k_norm_batch(const void *const *__restrict__ psis,
                                                         const int *__restrict__ Ns,
                                                         double *__restrict__ npart,
                                                         int *__restrict__ flags) {
    __shared__ double red[kThreads / 32];
    const int sidx = blockIdx.y;
    const v2_t<R> *psi = reinterpret_cast<const v2_t<R> *>(psis[sidx]);
    const uint64_t d = 1ull << Ns[sidx];
    double s = 0.0;
    int bad = 0;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < d;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const v2_t<R> v = psi[t];
        const double re = (double)v.x, im = (double)v.y;
        if (!isfinite(re) || !isfinite(im)) bad = 1;
        s += re * re + im * im;
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flags + sidx, kFlagNonFinite);
    const double b = block_sum(s, red);
    if (threadIdx.x == 0) npart[(size_t)sidx * gridDim.x + blockIdx.x] = b;
}

// M2 of every state of a batch: one warp per state, the same fixed-order
// segment sums as the single-state finalize (seg = {off1, n1, off2, n2}).
// status_out (may be null) receives each state's status with the same
// precedence as k_finalize: the batch's device-wait status first, then a
// non-finite amplitude, then a zero norm.
__global__ void k_finalize_batch(const longlong4 *__restrict__ seg, const double *__restrict__ parts,
                                 const double *__restrict__ npart, int nnorm,
                                 const int *__restrict__ flags, const int *__restrict__ Ns,
                                 const int *__restrict__ out_index, int count, const int *status,
                                 double *__restrict__ m2_out, int *__restrict__ status_out) {
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= count) return;
    const longlong4 g = seg[w];
    const double S = warp_sum_segments(parts, g.x, g.y, g.z, g.w);
    const double n = warp_sum_segments(npart, (long long)w * nnorm, nnorm, 0, 0);
    if ((threadIdx.x & 31) == 0) {
        int st = *status;
        if (st == 0 && (flags[w] & kFlagNonFinite)) st = SRE_ENONFINITE;
        if (st == 0 && !(n > 0.0)) st = SRE_EZERO;
        m2_out[out_index[w]] = m2_from(S, n, Ns[w], st != 0);
        if (status_out) status_out[out_index[w]] = st;
    }
}

template <typename R>
static size_t small_grid_for(const DeviceInfo &dev, int N, int S) {
    const uint64_t flat = (1ull << N) << (N - 1);
    const long long tps = (long long)((flat + kTile - 1) >> kTileBits);
    return (size_t)std::min<long long>(tps * S, (long long)dev.sms * 2);
}

BatchClass batch_class_layout(const DeviceInfo &dev, const Workspace &ws, int N, int S,
                              sre_mode_t mode, const LargeCfg *tuned_half, int tc_kind) {
    BatchClass L;
    L.tc_kind = tc_kind;
    L.N = N;
    L.S = S;
    const int eb = mode == SRE_MODE_FP64 ? 16 : 8;
    if (N <= kTileBits) {
        L.small_grid = (int)(eb == 8 ? small_grid_for<float>(dev, N, S) : small_grid_for<fx>(dev, N, S));
        const long long tps = (long long)((((1ull << N) << (N - 1)) + kTile - 1) >> kTileBits);
        L.cps_full = tps;  // tiles (= partials) per state
        L.parts_n = (size_t)S * (size_t)tps;
        return L;
    }
    const LargeCfg main = tuned_half ? *tuned_half : choose_main_cfg(dev, ws, N, mode, 1ull << N);
    L.two = takes_two(N, eb, tc_kind);
    if (one_applies(N, eb)) {
        // one partial per shift, all shifts or those below 4096 beside the
        // tensor-core kernel
        L.cfg_half = main;
        L.cps_full = tc_kind ? (long long)kTile : 0;
        L.cps_half = tc_kind ? (long long)((((1ull << N) - kTile) + (1ull << L.cfg_half.C_log) - 1) >> L.cfg_half.C_log)
                             : 1ll << N;
        L.parts_n = (size_t)S * (size_t)(L.cps_full + L.cps_half);
        L.chunks_max = tc_kind ? (size_t)S * (size_t)L.cps_half : 1;
        return L;
    }
    if (L.two) {
        // every shift in one launch, or the shifts below 4096 beside the
        // tensor-core kernel
        L.cfg_full = choose_two_cfg(dev, ws, N);
        L.cfg_half = L.cfg_full;
        if (tc_kind) L.cfg_half = main;
        L.cps_full = tc_kind ? two_layout(ws, L.cfg_full, N, 0, kTile).n_chunks : 0;
        L.cps_half = tc_kind ? (long long)((((1ull << N) - kTile) + (1ull << L.cfg_half.C_log) - 1) >> L.cfg_half.C_log)
                             : two_layout(ws, L.cfg_half, N, 0, 1ull << N).n_chunks;
        L.parts_n = (size_t)S * (size_t)(L.cps_full + L.cps_half);
        L.chunks_max = (size_t)S * (size_t)std::max(L.cps_full, L.cps_half);
        return L;
    }
    L.cfg_half = main;
    // the single-pass kernel has one partial per shift
    if (mid_applies(N, eb)) L.cfg_half.C_log = 0;
    L.cps_full = 0;
    L.cps_half = 1ll << (N - L.cfg_half.C_log);
    L.parts_n = L.chunks_max = (size_t)S * (size_t)L.cps_half;
    (void)ws;
    return L;
}

template <typename R>
static cudaError_t enqueue_batch_class_t(const Workspace &ws, const DeviceInfo &dev,
                                         const BatchClass &L, const void *const *d_ptrs,
                                         double *parts, unsigned *counters, size_t chunk_cap,
                                         cudaStream_t st, long long wait_ns, int *tc_e, double *tc_bn,
                                         size_t tc_cap) {
    cudaError_t e;
    const int N = L.N;
    if (N <= kTileBits) {
        int np = 0;
        e = launch_small<R>(N, nullptr, d_ptrs, L.S, 0, 1ull << N, parts + L.parts_off,
                            (int)L.parts_n, dev, st, &np, L.small_grid, 2);
        ws.launches += 1;
        return e;
    }
    size_t off = L.parts_off;
    for (int half = 0; half <= 1; ++half) {
        const LargeCfg &c = half ? L.cfg_half : L.cfg_full;
        const long long cps = half ? L.cps_half : L.cps_full;
        const uint64_t xb = half && L.cps_full ? (uint64_t)kTile : 0, xe = half ? (1ull << N) : (uint64_t)kTile;
        if constexpr (sizeof(cx_t<R>) == 8) {
            if (one_applies(N, 8) && !(half && L.tc_kind)) {
                if (cps == 0) continue;
                if ((e = cudaMemsetAsync(ws.work, 0, kWorkBytes, st)) != cudaSuccess) return e;
                if ((e = launch_one(N, nullptr, d_ptrs, L.S, 0, (uint64_t)cps, 2, parts + off, nullptr, ws.work + 2,
                                    ws.status, wait_ns, dev, st)) != cudaSuccess)
                    return e;
                ws.launches += 1;
                off += (size_t)cps * L.S;
                continue;
            }
            if (L.two && !(half && L.tc_kind)) {
                if (cps == 0) continue;
                if ((e = cudaMemsetAsync(counters, 0, sizeof(unsigned) * 3 * chunk_cap, st)) != cudaSuccess) return e;
                if ((e = cudaMemsetAsync(ws.work, 0, kWorkBytes, st)) != cudaSuccess) return e;
                if ((e = launch_two(ws, c, N, nullptr, d_ptrs, L.S, 0, half ? 1ull << N : (uint64_t)kTile, 2,
                                    parts + off, counters, chunk_cap, chunk_cap, ws.work + 2, nullptr, wait_ns, st)) !=
                    cudaSuccess)
                    return e;
                ws.launches += 1;
                off += (size_t)cps * L.S;
                continue;
            }
        }
        if (cps == 0) continue;
        if constexpr (sizeof(cx_t<R>) == 16) {
            if (mid_applies(N, 16)) {
                // one partial per shift
                if ((e = launch_mid(N, nullptr, d_ptrs, L.S, cps, 0, 2, parts + off, nullptr, dev, st)) != cudaSuccess)
                    return e;
                ws.launches += 1;
                off += (size_t)cps * L.S;
                continue;
            }
        }
        if (!large_cfg_fits(ws, c, N)) return cudaErrorInvalidValue;
        LargeArgs A;
        A.psi = nullptr;
        A.psis = d_ptrs;
        A.fx_exp = ws.fx_exp;
        A.fx_cap = ws.fx_cap;
        A.tc_e = tc_e;
        A.chunks_per_state = cps;
        A.N = N;
        A.h2 = N - kTileBits - 1;
        A.x_begin = xb;
        A.x_end = xe;
        A.x0 = xb;  // kTile and 0 are chunk-aligned
        A.C_log = c.C_log;
        A.R = c.R;
        A.G2_log = std::min(c.G2_log, A.h2);
        A.B1_log = std::max(0, std::min(c.B1_log, A.h2));
        A.stage1 = c.stage1;
        A.stage2 = c.stage2;
        A.alpha = 2;
        A.n_chunks = cps * L.S;
        A.D = (int)std::max<long long>(1, std::min<long long>(std::min(c.D, c.R - 1), A.n_chunks));
        A.P1 = 1 << (A.h2 - A.B1_log);
        A.P2 = (1 << c.C_log) << (A.h2 - A.G2_log);
        A.n_items = A.n_chunks * (long long)(A.P1 + A.P2);
        if ((size_t)A.n_chunks > chunk_cap || (size_t)A.R * A.P2 * 8 > ws.item_part_cap ||
            (sizeof(cx_t<R>) == 16 && (size_t)A.R << (A.C_log + A.h2) > ws.fx_cap))
            return cudaErrorInvalidValue;
        A.scratch = ws.scratch;
        A.item_part = ws.item_part;
        A.chunk_sum = parts + off;
        A.done1 = counters;
        A.done2 = counters + chunk_cap;
        A.freed = counters + 2 * chunk_cap;
        A.work = ws.work;
        A.per_x = nullptr;
        A.status = ws.status;
        A.wait_ns = wait_ns;
        if ((e = cudaMemsetAsync(counters, 0, sizeof(unsigned) * 3 * chunk_cap, st)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(ws.work, 0, sizeof(unsigned long long), st)) != cudaSuccess) return e;
        const int grid = (int)std::max<long long>(1, std::min<long long>(c.grid, A.n_items));
        if (half && L.tc_kind)
            e = launch_large_tc(A, ws, dev, grid, st, L.tc_kind, tc_e, tc_bn, tc_cap);
        else
            e = launch_large<R>(A, grid, st);
        if (e != cudaSuccess) return e;
        ws.launches += 1;
        off += (size_t)A.n_chunks;
    }
    return cudaSuccess;
}

cudaError_t enqueue_batch_class(const Workspace &ws, const DeviceInfo &dev, const BatchClass &L,
                                const void *const *d_ptrs, double *parts, unsigned *counters,
                                size_t chunk_cap, sre_mode_t mode, cudaStream_t st,
                                long long wait_ns, int *tc_e, double *tc_bn, size_t tc_cap) {
    if (mode == SRE_MODE_FP64)
        return enqueue_batch_class_t<fx>(ws, dev, L, d_ptrs, parts, counters, chunk_cap, st, wait_ns, tc_e,
                                         tc_bn, tc_cap);
    return enqueue_batch_class_t<float>(ws, dev, L, d_ptrs, parts, counters, chunk_cap, st, wait_ns, tc_e, tc_bn,
                                        tc_cap);
}

cudaError_t enqueue_batch_norm(const Workspace &ws, const void *const *d_ptrs, const int *d_Ns,
                               int count, double *npart, int *flags, sre_mode_t mode,
                               cudaStream_t st) {
    cudaError_t e;
    if ((e = cudaMemsetAsync(flags, 0, sizeof(int) * count, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ws.status, 0, sizeof(int), st)) != cudaSuccess) return e;
    const dim3 grid(kNormBlocks, count);
    if (mode == SRE_MODE_FP64)
        k_norm_batch<double><<<grid, kThreads, 0, st>>>(d_ptrs, d_Ns, npart, flags);
    else
        k_norm_batch<float><<<grid, kThreads, 0, st>>>(d_ptrs, d_Ns, npart, flags);
    ws.launches += 1;
    return cudaGetLastError();
}

cudaError_t enqueue_batch_finalize(const Workspace &ws, const void *seg, const double *parts,
                                   const double *npart, const int *flags, const int *d_Ns,
                                   const int *d_out_index, int count, double *m2_out,
                                   int *status_out, cudaStream_t st) {
    const int threads = 256;
    const int blocks = (count * 32 + threads - 1) / threads;
    k_finalize_batch<<<blocks, threads, 0, st>>>(reinterpret_cast<const longlong4 *>(seg), parts, npart,
                                                 kNormBlocks, flags, d_Ns, d_out_index, count,
                                                 ws.status, m2_out, status_out);
    ws.launches += 1;
    return cudaGetLastError();
}

cudaError_t enqueue_malpha_from_sums(const double *S, const double *n2, int N, int alpha, double *out,
                                     cudaStream_t st) {
    k_malpha_from_sums<<<1, 1, 0, st>>>(S, n2, N, alpha, out);
    return cudaGetLastError();
}

cudaError_t enqueue_convert(const void *src, sre_dtype_t from, void *dst, int N, cudaStream_t st) {
    const uint64_t d = 1ull << N;
    const int grid = (int)std::min<uint64_t>((d + kThreads - 1) / kThreads, 4096);
    if (from == SRE_C64)
        k_convert<double2, float2><<<grid, kThreads, 0, st>>>(reinterpret_cast<const float2 *>(src),
                                                              reinterpret_cast<double2 *>(dst), d);
    else
        k_convert<float2, double2><<<grid, kThreads, 0, st>>>(reinterpret_cast<const double2 *>(src),
                                                              reinterpret_cast<float2 *>(dst), d);
    return cudaGetLastError();
}

}  // namespace sre
