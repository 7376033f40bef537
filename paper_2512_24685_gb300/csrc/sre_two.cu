// sre_two.cu -- FP32 two-pass kernel for 17 <= N <= 19, all shifts in the
// halved form (sre_wht32.cuh); at N = 20 for the shifts below 4096 beside the
// tensor-core kernel.
//
// Pass 1 (one item: a block of 8192 entries for the 2^C_log shifts that share
// its factors) forms the products, transforms the 13 block bits and writes
// the block to a slot of a scratch ring as one row; pass 2 (one item: a set of
// columns of the rows) transforms the N - 14 row bits in registers and sums
// the powers.  In long ranges the factors of a block are loaded once per item into
// tensor memory: the item's shifts differ only in block bits that index registers, so
// each thread finds its own and its partner factors for all of them in its own
// tensor-memory columns, the partner's by an XOR of the column address, and
// the loads leave the L1 pipe.
//
// Shifts are grouped in chunks: 2^C_log shifts per item, 2^(13 - C_log) apart where
// they share factors (long ranges), else consecutive ones, times 2^U_log items
// per block (U_log > 0 where few blocks make a shift, so that a chunk has 16 items
// per pass or more).  A chunk owns one ring slot from its first
// pass-1 item to its last pass-2 item.
//
// What bounds it: about 30 SM cycles per 32 entries of the halved transform at
// N = 18, of which the transforms themselves take 20 (sre_one.cu); the rest are
// the row stores and loads through L2, the factor loads and the GPU-scope
// fence of each item.  DRAM carries 3.4 TB/s of ring traffic that L2 does not
// hold.  Measured on GB300: N = 18 109 ms for all shifts (16 entries per
// thread, 4096-entry blocks and a fixed item order: 196 ms), N = 19 50.6 ms for
// 58255 shifts (76.7 ms).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "sre_async.cuh"
#include "sre_internal.h"
#include "sre_two.h"
#include "sre_wht32.cuh"

namespace sre {
using namespace dev;

namespace {

constexpr int kPubWarp = 7;  // the warp that publishes finished items
constexpr int kTwoCtas = 2;  // CTAs per SM: 128 registers a thread, 64 KB and 256 tensor-memory columns each

struct TwoArgs {
    const float2 *psi;
    const void *const *psis;
    long long chunks_per_state;
    int N;
    uint64_t x_begin, x_end, x0;
    int W_log, C_log, U_log, R;
    int alpha;
    long long n_chunks;
    float2 *scratch;
    double *item_part, *chunk_sum;
    // per chunk: finished items of both passes; the pass-2 order (chunk + 1);
    // the ring slot the chunk takes (slot + 1, chunks from R up)
    unsigned *done, *ready, *slot_of;
    unsigned char *work;  // counters, one 128-byte line each (TwoCounter)
    double *per_x;
    int *status;
    long long wait_ns;
};

// Spacing (log2) of an item's shifts, and of a chunk's shifts in other items.
template <bool SHARE>
__device__ __forceinline__ int two_spacing(const TwoArgs &a) { return SHARE ? kBlockBits - a.C_log : 0; }
template <bool SHARE>
__device__ __forceinline__ int two_item_spacing(const TwoArgs &a) { return SHARE ? 0 : a.C_log; }

__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

constexpr int kRowReals = 2 << kBlockBits;  // real columns of a scratch row (64 KB)

// A thread transforms 64 real values of a shift's scratch rows: V = 64 / 2^H2
// columns of all 2^H2 rows.
template <int H2>
struct TwoCols {
    static constexpr int V = 64 >> H2;
    static constexpr int kWarpCols = 32 * V;  // columns of one warp's unit
    static constexpr int kParts = 8;          // partials of an item and shift (one per warp)
};

// 2^H2-point transforms of the columns at `col` (the lane's first) and the
// sum of powers over them.
template <int H2>
__device__ __forceinline__ double two_columns(const float *col, int alpha) {
    constexpr int V = TwoCols<H2>::V;
    c64_t v[32];
    if constexpr (V == 1) {
        // one real column: rows r and r ^ 4 share a packed register, so that
        // row bit 2 is transformed inside it
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int r = (i & 3) | ((i >> 2) << 3);
            v[i] = Cx<float>::pack(__ldcg(col + (size_t)r * kRowReals), __ldcg(col + (size_t)(r | 4) * kRowReals));
        }
        w32_stage<2>(v);  // row bits 3, 4, 5
        w32_stage<3>(v);
        w32_stage<4>(v);
        w32_stage<0>(v);  // row bits 0, 1
        w32_stage<1>(v);
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            float a, b;
            Cx<float>::unpack(v[i], a, b);
            v[i] = Cx<float>::pack(a + b, a - b);
        }
    } else {
        // v[r * V / 2 + p]: columns 2 p, 2 p + 1 of row r
        constexpr int P = V / 2, PL = 5 - H2;
#pragma unroll
        for (int r = 0; r < (1 << H2); ++r) {
            if constexpr (V == 2) {
                v[r] = __ldcg(reinterpret_cast<const unsigned long long *>(col + (size_t)r * kRowReals));
            } else {
#pragma unroll
                for (int p = 0; p < P; p += 2) {
                    const ulonglong2 q = __ldcg(reinterpret_cast<const ulonglong2 *>(col + (size_t)r * kRowReals + 2 * p));
                    v[r * P + p] = q.x;
                    v[r * P + p + 1] = q.y;
                }
            }
        }
        if constexpr (H2 > 3) w32_stage<PL + 3>(v);
        if constexpr (H2 > 4) w32_stage<PL + 4>(v);
        w32_stage<PL + 0>(v);
        w32_stage<PL + 1>(v);
        w32_stage<PL + 2>(v);
    }
    return w32_pow(v, alpha);
}

// ------------------------------------------------------------- scheduling
//
// Items are handed out as they become possible, never waited for: a pass-1
// item once its chunk has a free ring slot, a pass-2 item once its chunk's
// pass 1 is complete.  Chunks become ready, and slots free, in any order; two
// lists keep that order, and a pair of credit counters says how many items
// may be claimed (a claim takes a credit, then a ticket, so a ticket always
// points at something published or about to be).  Pass 2 goes first, which
// keeps the ring small.  Handing items out in a fixed order with a lag between
// the passes made CTAs wait a quarter of the time even with a ring twice the
// size: items of one chunk end far apart, because the warps of an SM do not
// progress evenly.
enum TwoCounter { kCredits, kTick1, kTick2, kReadyCount, kFreedCount };

template <typename T>
__device__ __forceinline__ T *two_counter(const TwoArgs &a, TwoCounter k) {
    return reinterpret_cast<T *>(a.work + 128 * (int)k);
}

struct TwoItem {
    long long c;  // chunk; -1: none yet, -2: no more items
    int r;        // item of the chunk's pass
    int slot, pass1;
};

// One lane's claim, advanced in steps so that each access's latency passes
// behind the tile work between two steps: read both credits, take one, take a
// ticket.  The read comes first because a refused claim takes its credit for
// a moment: hundreds of idle CTAs asking blindly would keep the counter below
// zero whatever is added to it.
struct TwoClaim {
    int st = 0;  // 0 idle, 1 credits read, 2 / 4 credit of pass 2 / 1 asked, 3 / 5 ticket asked
    int v1 = 0, v2 = 0;
    long long i = 0;
};

__device__ __forceinline__ void two_step(const TwoArgs &a, TwoClaim &k, int P_log) {
    int *credit = two_counter<int>(a, kCredits);  // pass 1, pass 2
    // pass 1 counts from zero: the first R chunks are possible at once
    const int first = (int)(min((long long)a.R, a.n_chunks) << P_log);
    switch (k.st) {
        case 0:
            asm volatile("ld.relaxed.gpu.global.v2.s32 {%0, %1}, [%2];"
                         : "=r"(k.v1), "=r"(k.v2)
                         : "l"(credit)
                         : "memory");
            k.st = 1;
            break;
        case 1:
            if (k.v2 > 0) {
                k.v2 = atomicSub(credit + 1, 1);
                k.st = 2;
            } else if (k.v1 + first > 0) {
                k.v1 = atomicSub(credit, 1);
                k.st = 4;
            } else {
                k.st = 0;
            }
            break;
        case 2:
            if (k.v2 > 0) {
                k.i = (long long)atomicAdd(two_counter<unsigned long long>(a, kTick2), 1ull);
                k.st = 3;
            } else {
                atomicAdd(credit + 1, 1);
                k.st = 0;
            }
            break;
        case 4:
            if (k.v1 + first > 0) {
                k.i = (long long)atomicAdd(two_counter<unsigned long long>(a, kTick1), 1ull);
                k.st = 5;
            } else {
                atomicAdd(credit, 1);
                k.st = 0;
            }
            break;
        default: break;
    }
}

// The claimed item if the claim is complete (its list entry may still be on
// its way), else c = -1.
__device__ __forceinline__ TwoItem two_take(const TwoArgs &a, TwoClaim &k, int P_log) {
    TwoItem t;
    t.c = -1;
    const long long pos = k.i >> P_log;
    t.r = (int)(k.i & ((1ll << P_log) - 1));
    if (k.st == 3) {
        const unsigned e = ld_acquire_u32(a.ready + pos);
        if (!e) return t;
        t.pass1 = 0;
        t.c = (long long)e - 1;
        t.slot = t.c < a.R ? (int)t.c : (int)__ldcg(a.slot_of + t.c) - 1;
        k.st = 0;
    } else if (k.st == 5) {
        unsigned e = 0;
        if (pos >= a.R && !(e = ld_acquire_u32(a.slot_of + pos))) return t;
        t.pass1 = 1;
        t.c = pos;
        t.slot = pos < a.R ? (int)pos : (int)e - 1;
        k.st = 0;
    }
    return t;
}

// Claims until there is an item, no more work, an error, or the time limit
// (SRE_ETIMEDOUT).
__device__ __noinline__ TwoItem two_claim(const TwoArgs &a, TwoClaim k, int P_log) {
    const unsigned long long t0 = globaltimer_ns();
    TwoItem t;
    for (unsigned it = 0; it < (1u << 28); ++it) {
        two_step(a, k, P_log);
        t = two_take(a, k, P_log);
        if (t.c >= 0) return t;
        if (k.st == 1 || k.st == 2 || k.st == 4) continue;
        // nothing possible, or the ticket's list entry is on its way
        t.c = -2;
        if (*(volatile int *)a.status != 0) return t;
        if (k.st == 0 && *two_counter<volatile unsigned long long>(a, kTick2) >=
                             (unsigned long long)a.n_chunks << P_log)
            return t;
        if ((long long)(globaltimer_ns() - t0) > a.wait_ns) break;
        __nanosleep(100);
    }
    atomicCAS(a.status, 0, (int)SRE_ETIMEDOUT);
    t.c = -2;
    return t;
}

// A finished item that has not been published yet.  Publishing costs a
// GPU-scope fence, which waits for the CTA's scratch stores; done at once it
// would hold all warps at their next barrier, so one warp does it in the
// middle of the next item, when the stores have drained -- or before the CTA
// waits for an item, since that may depend on its own unpublished one.
struct TwoDone {
    TwoItem t;    // t.c = -1: none
    uint64_t xc;  // the chunk's first shift
};

template <int H2, bool SHARE>
__device__ __noinline__ void two_publish(const TwoArgs &a, TwoDone *d) {
    const int lane = threadIdx.x & 31, C = 1 << a.C_log, S_log = a.C_log + a.U_log, P_log = H2 + a.U_log;
    const long long c = d->t.c;
    if (c < 0) return;
    unsigned old = 0;
    if (lane == 0) {
        fence_gpu();
        old = atomicAdd(a.done + c, 1u) + 1;
        if (old == 1u << P_log) {
            // pass 1 complete: pass 2 of the chunk becomes possible
            fence_gpu();
            const unsigned at = atomicAdd(two_counter<unsigned>(a, kReadyCount), 1u);
            atomicExch(a.ready + at, (unsigned)c + 1);
            fence_gpu();
            atomicAdd(two_counter<int>(a, kCredits) + 1, 1 << P_log);
        }
    }
    old = __shfl_sync(0xffffffffu, old, 0);
    if (old == 2u << P_log) {
        // last item of the chunk: per-shift and chunk sums in fixed order
        fence_gpu();
        constexpr int kParts = TwoCols<H2>::kParts;
        double cs = 0.0;
        for (int q = 0; q < (1 << S_log); ++q) {
            const double *ip = a.item_part + (((((size_t)d->t.slot << S_log) + q) << H2) * kParts);
            double sx = 0.0;
            for (int m = lane; m < (kParts << H2); m += 32) sx += __ldcg(ip + m);
            const uint64_t x = d->xc + ((uint64_t)(q >> a.C_log) << two_item_spacing<SHARE>(a)) +
                               ((uint64_t)(q & (C - 1)) << two_spacing<SHARE>(a));
            sx = fp32_scale(fp32_doubled(x), a.alpha) * warp_sum(sx);
            if (lane == 0 && a.per_x && x >= a.x_begin && x < a.x_end) a.per_x[x - a.x_begin] = sx;
            cs += sx;
        }
        if (lane == 0) {
            a.chunk_sum[c] = cs;
            // the slot goes to the next chunk without one
            fence_gpu();
            const long long to = a.R + (long long)atomicAdd(two_counter<unsigned>(a, kFreedCount), 1u);
            if (to < a.n_chunks) {
                atomicExch(a.slot_of + to, (unsigned)d->t.slot + 1);
                fence_gpu();
                atomicAdd(two_counter<int>(a, kCredits), 1 << P_log);
            }
        }
    }
    __syncwarp();
    if (lane == 0) d->t.c = -1;
    __syncwarp();
}

template <int H2, bool SHARE>
__global__ void __launch_bounds__(kBlockThreads, kTwoCtas) k_two(const __grid_constant__ TwoArgs a) {
    extern __shared__ __align__(1024) unsigned char buf[];
    __shared__ TwoItem s_next;
    __shared__ TwoDone s_done;
    __shared__ uint32_t s_tmem;
    using Cols = TwoCols<H2>;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int C = 1 << a.C_log, S_log = a.C_log + a.U_log;
    const int P_log = H2 + a.U_log;  // items per chunk and pass

    if (SHARE && warp == 0) tc_alloc(&s_tmem, 2 * kFactorCols);
    TwoClaim claim;  // thread 0
    if (tid == 0) {
        s_done.t.c = -1;
        s_next = two_claim(a, claim, P_log);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // this warp's 32 lanes; warps w and w + 4 share them
    const uint32_t tmem = SHARE ? s_tmem + ((uint32_t)(warp & 3) << 21) + (warp >> 2) * kFactorCols : 0;
    while (s_next.c >= 0) {
        const long long c = s_next.c;
        const int r = s_next.r, slot = s_next.slot;
        const bool pass1 = s_next.pass1 != 0;
        long long cl = c;
        const float2 *psi = a.psi;
        if (a.psis) {
            const long long sidx = c / a.chunks_per_state;
            cl = c - sidx * a.chunks_per_state;
            psi = reinterpret_cast<const float2 *>(a.psis[sidx]);
        }
        // chunk cl: shifts k < 2^C_log of items u < 2^U_log, from xc
        const int cw_log = a.W_log - S_log, u = r >> H2, b = r & ((1 << H2) - 1);
        const uint64_t xc = a.x0 + ((uint64_t)(cl >> cw_log) << a.W_log) +
                            ((uint64_t)(cl & ((1ll << cw_log) - 1)) << a.U_log);
        const uint64_t x0 = xc + ((uint64_t)u << two_item_spacing<SHARE>(a));
        // the item's first scratch row block
        float2 *base = a.scratch + ((((((size_t)slot << a.U_log) + (size_t)u) << a.C_log)) << (H2 + kBlockBits));
        if (pass1) {
            bool filled = false;
            for (int k = 0; k < C; ++k) {
                const uint64_t x = x0 + ((uint64_t)k << two_spacing<SHARE>(a));
                const bool claiming = tid == 0 && k + 1 == C;
                if (claiming) two_step(a, claim, P_log);
                __syncwarp();
                if (x < a.x_begin || x >= a.x_end) continue;
                // from x = 8192 up the item's shifts share the pivot and differ
                // in register bits alone: one fill serves them all.  A shift
                // that shares nothing takes its factors straight to registers
                c64_t v[32];
                if (SHARE && x >= (1u << kBlockBits)) {
                    if (!filled) w32_fill(tmem, pair_src(psi, a.N, x0, b), tid);
                    filled = true;
                    if (warp == kPubWarp) two_publish<H2, SHARE>(a, &s_done);
                    w32_products(v, tmem, (uint32_t)k << (3 - a.C_log));
                } else {
                    if (warp == kPubWarp) two_publish<H2, SHARE>(a, &s_done);
                    w32_direct<0, 32>(v, pair_src(psi, a.N, x, b), tid);
                }
                if (claiming) two_step(a, claim, P_log);
                __syncwarp();
                w32_block(v, buf, tid);
                if (claiming) two_step(a, claim, P_log);
                __syncwarp();
                // entry order inside a row is free (pass 2 sums over it):
                // register-major, so that a warp stores 256-byte runs
                unsigned long long *o = reinterpret_cast<unsigned long long *>(
                                            base + ((size_t)k << (H2 + kBlockBits)) + ((size_t)b << kBlockBits)) +
                                        tid;
#pragma unroll
                for (int i = 0; i < 32; ++i) __stcg(o + (i << 8), v[i]);
                if (claiming) two_step(a, claim, P_log);
                __syncwarp();
            }
        } else {
            const int wc = (b * Cols::kParts + warp) * Cols::kWarpCols;
            for (int k = 0; k < C; ++k) {
                const uint64_t x = x0 + ((uint64_t)k << two_spacing<SHARE>(a));
                const bool claiming = tid == 0 && k + 1 == C;
                if (claiming) two_step(a, claim, P_log);
                __syncwarp();
                double s = 0.0;
                if (x >= a.x_begin && x < a.x_end) {
                    const float *cols = reinterpret_cast<const float *>(base + ((size_t)k << (H2 + kBlockBits))) + wc;
                    s = two_columns<H2>(cols + lane * Cols::V, a.alpha);
                    if (claiming) two_step(a, claim, P_log);
                    __syncwarp();
                    if (warp == kPubWarp) two_publish<H2, SHARE>(a, &s_done);
                    s = warp_sum(s);
                    if (claiming) two_step(a, claim, P_log);
                    __syncwarp();
                    // the unit's 128-byte lines have been read for the last
                    // time: drop them from L2 before they are written back
#pragma unroll
                    for (int m = 0; m < (Cols::V << H2) / 32; ++m) {
                        const int L = m * 32 + lane;  // V lines of each row
                        discard_l2_line(cols + (size_t)(L / Cols::V) * kRowReals + (L % Cols::V) * 32);
                    }
                    if (claiming) two_step(a, claim, P_log);
                    __syncwarp();
                }
                if (lane == 0) {
                    const size_t q = (((((size_t)slot << a.U_log) + u) << a.C_log) + k) << H2;
                    a.item_part[(q + b) * Cols::kParts + warp] = s;
                }
            }
        }
        if (warp == kPubWarp) two_publish<H2, SHARE>(a, &s_done);  // an item without work has not come by it
        __syncthreads();
        if (warp == kPubWarp && lane == 0) {
            s_done.t.c = c;
            s_done.t.slot = slot;
            s_done.xc = xc;
        }
        if (tid == 0) s_next = two_take(a, claim, P_log);
        __syncthreads();
        if (s_next.c == -1) {
            if (warp == kPubWarp) two_publish<H2, SHARE>(a, &s_done);
            TwoItem t;
            if (tid == 0) {
                t = two_claim(a, claim, P_log);
                claim = TwoClaim();
            }
            __syncthreads();  // every thread has seen that there was none
            if (tid == 0) s_next = t;
            __syncthreads();
        }
    }
    if (warp == kPubWarp) two_publish<H2, SHARE>(a, &s_done);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (SHARE && warp == 0) tc_dealloc(s_tmem, 2 * kFactorCols);
}

template <int H2>
cudaError_t launch_two_h(const TwoArgs &a, bool share, int grid, cudaStream_t st) {
    auto kern = share ? k_two<H2, true> : k_two<H2, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMoveBytes);
    if (e != cudaSuccess) return e;
    kern<<<grid, kBlockThreads, kMoveBytes, st>>>(a);
    return cudaGetLastError();
}

int two_h2(int N) { return N - 1 - kBlockBits; }
int two_u_log(int N) { return std::max(0, 4 - two_h2(N)); }

}  // namespace

bool two_applies(int N, int elem_bytes) { return elem_bytes == 8 && N >= 17 && N <= 20; }

// The kernel takes no tuning of the caller's: the fields were found for kernels
// with other items (a ring of chunks and a lag between the passes), and read as
// its own they cost up to 45 % (N = 20, one shift per item: no factors shared).
// Four shifts per item share one fill of the factors; the ring takes the
// workspace's tuning scratch (192 MB), less where the workspace has less.  With
// a ring that fits L2 the CTAs run out of slots: a chunk lives for two item
// times and the spread between its first and last item, and 304 CTAs hold 4
// shifts of 64 KB each.  N = 18, 16384 shifts: 7.0 ms with 192 MB, 10.1 ms
// with 96 MB, 14.1 ms with 64 MB; two shifts per item 8.3 ms at 128 MB.
LargeCfg choose_two_cfg(const DeviceInfo &dev, const Workspace &ws, int N) {
    LargeCfg c;
    c.C_log = 2;
    c.G2_log = 0;
    c.B1_log = 0;
    c.grid = std::max(1, dev.sms * kTwoCtas);
    while (c.C_log > 0 && ws.scratch_bytes >> c.C_log < (size_t)64 << (N - 1)) --c.C_log;  // 8 slots at least
    const size_t chunk = (size_t)8 << (c.C_log + two_u_log(N) + N - 1);
    c.R = (int)std::max<size_t>(2, std::min<size_t>(kMaxRing, std::min(ws.scratch_bytes, kTuneScratch) / chunk));
    c.D = 1;  // not used: items are handed out as they become possible
    return c;
}

namespace {
// Does the configuration fit the workspace (ring of scratch, item partials)?
bool two_fits(const Workspace &ws, const LargeCfg &c, int N, int U_log) {
    const size_t ring = (size_t)c.R << (c.C_log + U_log + N - 1 + 3);
    const size_t parts = (size_t)c.R << (c.C_log + U_log + two_h2(N) + 3);
    return ring <= ws.scratch_bytes && parts <= ws.item_part_cap;
}
}  // namespace

TwoLayout two_layout(const Workspace &ws, const LargeCfg &c, int N, uint64_t xb, uint64_t xe) {
    TwoLayout L;
    L.U_log = two_u_log(N);
    while (L.U_log > 0 && !two_fits(ws, c, N, L.U_log)) --L.U_log;
    // Windows of 8192 shifts whose items share factors; a shorter range would
    // leave most of a window empty and takes consecutive shifts, which share no
    // factors but a claim and a publication per item (N = 17, us for 2048 and
    // 8192 shifts: 575 and 2054; one shift per item: 769 and 2940; the general
    // kernel: 677 and 2551), fewer of them where the items run out.
    const uint64_t n = xe - xb;
    L.share = n >= 16384 && c.C_log > 0;
    L.C_log = n >= 1024 ? c.C_log : n >= 256 ? std::min(c.C_log, 1) : 0;
    L.R = c.R << (c.C_log - L.C_log);
    L.W_log = L.share ? kBlockBits : L.C_log + L.U_log;
    L.x0 = xb & ~((1ull << L.W_log) - 1);
    const uint64_t windows = (xe - L.x0 + (1ull << L.W_log) - 1) >> L.W_log;
    L.n_chunks = (long long)(windows << (L.W_log - L.C_log - L.U_log));
    return L;
}

cudaError_t launch_two(const Workspace &ws, const LargeCfg &c, int N, const void *psi, const void *const *psis,
                       int nstates, uint64_t xb, uint64_t xe, int alpha, double *chunk_sum, unsigned *counters,
                       size_t counter_stride, size_t counter_cap, unsigned long long *work, double *per_x,
                       long long wait_ns, cudaStream_t st) {
    if (!two_fits(ws, c, N, 0)) return cudaErrorInvalidValue;
    const TwoLayout L = two_layout(ws, c, N, xb, xe);
    TwoArgs a;
    a.psi = reinterpret_cast<const float2 *>(psi);
    a.psis = psis;
    a.chunks_per_state = L.n_chunks;
    a.N = N;
    a.x_begin = xb;
    a.x_end = xe;
    a.x0 = L.x0;
    a.W_log = L.W_log;
    a.C_log = L.C_log;
    a.U_log = L.U_log;
    a.R = L.R;
    a.n_chunks = L.n_chunks * nstates;
    if ((size_t)a.n_chunks > counter_cap) return cudaErrorInvalidValue;
    a.alpha = alpha;
    const long long n_items = a.n_chunks << (two_h2(N) + L.U_log + 1);
    a.scratch = reinterpret_cast<float2 *>(ws.scratch);
    a.item_part = ws.item_part;
    a.chunk_sum = chunk_sum;
    a.done = counters;
    a.ready = counters + counter_stride;
    a.slot_of = counters + 2 * counter_stride;
    a.work = reinterpret_cast<unsigned char *>(work);
    a.per_x = per_x;
    a.status = ws.status;
    a.wait_ns = wait_ns;
    const int grid = (int)std::max<long long>(1, std::min<long long>(c.grid, n_items));
    switch (two_h2(N)) {
        case 3: return launch_two_h<3>(a, L.share, grid, st);
        case 4: return launch_two_h<4>(a, L.share, grid, st);
        case 5: return launch_two_h<5>(a, L.share, grid, st);
        case 6: return launch_two_h<6>(a, L.share, grid, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace sre
