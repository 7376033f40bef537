// sre_wht32.cuh -- 13-bit Walsh-Hadamard transform of an 8192-entry block by
// 256 threads, 32 complex FP32 entries each, for conjugate-symmetry halved
// shifts.
//
// Halving holds for every shift x >= 1 with pivot j = the highest set bit of
// x: the transform W of g_x restricted to t_j = 0 runs over the N - 1 bit
// index t' (t with bit j removed) and sum_z |A_x(z)|^(2 alpha) =
// 2^(2 alpha) sum_z' [(Re W)^(2 alpha) + (Im W)^(2 alpha)].  The shift x = 0
// (g real) takes the same form: with g0, g1 the halves of g_0 by its top bit,
// W := transform of ((g0 + g1) + i (g0 - g1)) / 2 has A_0 = 2 Re W and 2 Im W.
//
// A block is the 8192 entries with the same high bits of t' (for N < 14 it
// holds 2^(14 - N) whole shifts).  Layouts (thread bits: lane 0-4, warp 5-7;
// register bits 0-4), e = entry index in the block:
//   round 1: thread = e0 e1 e2 e3 e5 | e6 e7 e8, register = e4 e9 e10 e11 e12
//   round 2: thread = e2 e3 e9 e10 e5 | e4 e11 e12, register = e0 e1 e6 e7 e8
// Round 1 transforms its five register bits, then the block moves once
// through shared memory (entry (i, tau) at slot (i << 8) | (tau ^ (i >> 1 & 3)):
// 16 distinct bank pairs per half-warp on both sides), round 2 transforms its
// five register bits, and the three bits left in lanes (e2, e3, e5) follow by
// half-exchanges: a lane pair swaps the upper half of a register bit that is
// already transformed, so that both values of the lane bit meet in one thread
// at one shuffle per entry.  The stage of that register bit writes sum and
// difference in swapped order in the upper lane (a multiply-add by +-1), which
// makes the swap the same instruction in both lanes; the signs this leaves on
// some outputs are the same for every block of a shift and vanish in the even
// powers.  Against 16 entries per thread (two moves per 12 bits) the block
// costs one move and three shuffles per 13 bits.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "sre_tc.cuh"
#include "sre_tile.cuh"

namespace sre {
namespace dev {

using c64_t = cx_t<float>;
constexpr int kBlockBits = 13;
constexpr int kBlockThreads = 256;
constexpr int kMoveBytes = 8192 * 8;    // move buffer of one block
constexpr uint32_t kFactorCols = 128;   // tensor-memory columns of a warp: own 64, partner 64

// entry bits of a round-1 register index and of a round-1 thread index
__host__ __device__ constexpr int w32_reg(int i) { return ((i & 1) << 4) | ((i >> 1) << 9); }
__host__ __device__ constexpr int w32_thr(int t) { return (t & 15) | ((t >> 4) << 5); }

// Butterflies over register bit B.
template <int B>
__device__ __forceinline__ void w32_stage(c64_t (&v)[32]) {
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        if (!(i & (1 << B))) {
            const c64_t a = v[i], b = v[i | (1 << B)];
            v[i] = Cx<float>::add(a, b);
            v[i | (1 << B)] = Cx<float>::sub(a, b);
        }
    }
}

// The same with sum and difference in swapped order where s = -1.
template <int B>
__device__ __forceinline__ void w32_stage_signed(c64_t (&v)[32], float s) {
    const c64_t p = Cx<float>::pack(s, s), m = Cx<float>::pack(-s, -s);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        if (!(i & (1 << B))) {
            const c64_t a = v[i], b = v[i | (1 << B)];
            v[i] = Cx<float>::fma(b, p, a);
            v[i | (1 << B)] = Cx<float>::fma(b, m, a);
        }
    }
}

// Swap the upper half of register bit B with the lane across `mask`, then the
// butterflies over the lane bit.
template <int B>
__device__ __forceinline__ void w32_lane_stage(c64_t (&v)[32], int mask) {
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        if (!(i & (1 << B))) {
            const c64_t a = v[i], r = __shfl_xor_sync(0xffffffffu, v[i | (1 << B)], mask);
            v[i] = Cx<float>::add(a, r);
            v[i | (1 << B)] = Cx<float>::sub(a, r);
        }
    }
}

// Keeps what is derived from x from being computed once outside the caller's
// loop, where it would stay live beside the data registers.
__device__ __forceinline__ uint32_t local_copy(uint32_t x) {
    asm volatile("" : "+r"(x));
    return x;
}

// Transform over the block bits below NB (12 or 13): round 1, move, round
// 2.  HALF moves real and imaginary parts one after the other through a buffer
// of half the size.
template <int NB = kBlockBits, bool HALF = false>
__device__ __forceinline__ void w32_block(c64_t (&v)[32], unsigned char *buf, int tid) {
    w32_stage<1>(v);
    w32_stage<2>(v);
    w32_stage<3>(v);
    if constexpr (NB > 12) w32_stage<4>(v);
    w32_stage<0>(v);
    const int tau = (int)local_copy((uint32_t)tid);
    // round-1 register index and slot bits of this thread's round-2 entries
    const int i2 = ((tau >> 5) & 1) | (((tau >> 2) & 3) << 1) | ((tau >> 6) << 3);
    const int f = (tau >> 2) & 3;
    if constexpr (!HALF) {
        __syncthreads();  // the previous block's readers are done
#pragma unroll
        for (int i = 0; i < 32; ++i)
            *reinterpret_cast<c64_t *>(buf + (i << 11) + ((tau ^ ((i >> 1) & 3)) << 3)) = v[i];
        __syncthreads();
        const unsigned char *row = buf + (i2 << 11) + ((tau & 3) << 5) + (((tau >> 4) & 1) << 7);
#pragma unroll
        for (int k = 0; k < 32; ++k)
            v[k] = *reinterpret_cast<const c64_t *>(row + ((k >> 2) << 8) + (((k & 3) ^ f) << 3));
    } else {
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                float p[2];
                Cx<float>::unpack(v[i], p[0], p[1]);
                *reinterpret_cast<float *>(buf + (i << 10) + ((tau ^ ((i >> 1) & 3)) << 2)) = p[part];
            }
            __syncthreads();
            const unsigned char *row = buf + (i2 << 10) + ((tau & 3) << 4) + (((tau >> 4) & 1) << 6);
#pragma unroll
            for (int k = 0; k < 32; ++k) {
                float p[2];
                Cx<float>::unpack(v[k], p[0], p[1]);
                p[part] = *reinterpret_cast<const float *>(row + ((k >> 2) << 7) + (((k & 3) ^ f) << 2));
                v[k] = Cx<float>::pack(p[0], p[1]);
            }
        }
    }
    w32_stage<3>(v);
    w32_stage<4>(v);
    w32_stage_signed<2>(v, (tau & 16) ? -1.f : 1.f);
    w32_stage_signed<0>(v, (tau & 2) ? -1.f : 1.f);
    w32_stage_signed<1>(v, (tau & 1) ? -1.f : 1.f);
    w32_lane_stage<1>(v, 1);
    w32_lane_stage<0>(v, 2);
    w32_lane_stage<2>(v, 16);
}

// -------------------------------------------------------------- factors

// Where one shift finds the factors of a block: own entry at byte offset o
// from `own`, its partner t ^ x at offset o ^ xo from `par`.  pivot < 13: the
// entry bits from the pivot up sit one place higher in t.
struct PairSrc {
    const unsigned char *own, *par;
    uint32_t xo;
    int pivot;   // kBlockBits: the pivot lies above the block
    bool zero;   // x = 0
    bool twice;  // fp32_doubled
};

__device__ __forceinline__ PairSrc pair_src(const float2 *psi, int N, uint64_t x, int tp) {
    PairSrc s;
    s.zero = x == 0;
    s.twice = fp32_doubled(x);
    const uint64_t xe = s.zero ? 1ull << (N - 1) : x;  // x = 0 pairs the two halves
    const int j = 63 - __clzll((long long)xe);
    if (j >= kBlockBits) {
        const int jh = j - kBlockBits;
        const uint64_t th = (((uint64_t)tp >> jh) << (jh + 1)) | ((uint64_t)tp & ((1ull << jh) - 1));
        s.own = reinterpret_cast<const unsigned char *>(psi + (th << kBlockBits));
        s.par = reinterpret_cast<const unsigned char *>(psi + ((th ^ (xe >> kBlockBits)) << kBlockBits));
        s.xo = (uint32_t)(xe & ((1u << kBlockBits) - 1)) << 3;
        s.pivot = kBlockBits;
    } else {
        s.own = s.par = reinterpret_cast<const unsigned char *>(psi + ((uint64_t)tp << (kBlockBits + 1)));
        s.xo = (uint32_t)xe << 3;
        s.pivot = j;
    }
    return s;
}

__device__ __forceinline__ void tmem_ld8(uint32_t addr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(addr)
                 : "memory");
}

// Completes the loads of p and q: their registers pass through, so that no
// use of them moves ahead of the wait.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&p)[8], uint32_t (&q)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(p[0]), "+r"(p[1]), "+r"(p[2]), "+r"(p[3]), "+r"(p[4]), "+r"(p[5]), "+r"(p[6]), "+r"(p[7]),
                   "+r"(q[0]), "+r"(q[1]), "+r"(q[2]), "+r"(q[3]), "+r"(q[4]), "+r"(q[5]), "+r"(q[6]), "+r"(q[7])::
                     "memory");
}

// Byte offset of entry bits e of a block in t, for the pivot of s (linear in
// the bits of e).
__device__ __forceinline__ uint32_t w32_place(const PairSrc &s, int e) {
    if (s.pivot == kBlockBits) return (uint32_t)e << 3;
    const int lo = e & ((1 << s.pivot) - 1);
    return (uint32_t)((((e - lo) << 1) | lo) << 3);
}

// x = 0: the value of W's input from the two halves of g_0.
__device__ __forceinline__ float2 w32_zero_value(float2 a, float2 b) {
    const float g0 = a.x * a.x + a.y * a.y, g1 = b.x * b.x + b.y * b.y;
    return make_float2(0.5f * (g0 + g1), 0.5f * (g0 - g1));
}

template <int F, int COUNT>
__device__ __forceinline__ void w32_double(c64_t (&v)[32]) {
#pragma unroll
    for (int i = F; i < F + COUNT; ++i) v[i] = Cx<float>::add(v[i], v[i]);
}

// Products of the entries with register index [F, F + COUNT) (and the thread's
// bits), by loads of both factors, doubled where the shift asks for it (TWICE).
template <int F, int COUNT, bool TWICE = true>
__device__ __forceinline__ void w32_direct(c64_t (&v)[32], const PairSrc &s, int tid) {
    const int tau = (int)local_copy((uint32_t)tid);
    const uint32_t o = w32_place(s, w32_thr(tau));
    uint32_t w[5];
#pragma unroll
    for (int b = 0; b < 5; ++b) w[b] = w32_place(s, w32_reg((1 << b) & (COUNT - 1)));
#pragma unroll
    for (int i = 0; i < COUNT; ++i) {
        uint32_t oi = o;
#pragma unroll
        for (int b = 0; b < 5; ++b)
            if (i & (1 << b)) oi += w[b];
        const float2 a = __ldg(reinterpret_cast<const float2 *>(s.own + oi));
        const float2 b = __ldg(reinterpret_cast<const float2 *>(s.par + (oi ^ s.xo)));
        if (s.zero) {
            const float2 z = w32_zero_value(a, b);
            v[F + i] = Cx<float>::pack(z.x, z.y);
        } else {
            v[F + i] = conj_mul<float>(b.x, b.y, a.x, a.y);  // conj(phi_{t^x}) * phi_t
        }
    }
    if (TWICE && s.twice) w32_double<F, COUNT>(v);
}

__device__ __forceinline__ void tmem_put4(uint32_t addr, const c64_t *v) {
    uint32_t r[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        r[2 * q] = (uint32_t)v[q];
        r[2 * q + 1] = (uint32_t)(v[q] >> 32);
    }
    tc_st8(addr, r);
}

// Load the own and partner factors of one block, for a shift with the pivot above
// it, into this thread's tensor-memory columns (own entry i at columns 2i, partner
// at 64 + 2i).
__device__ __forceinline__ void w32_fill(uint32_t tmem, const PairSrc &s, int tid) {
    const int tau = (int)local_copy((uint32_t)tid);
    const uint32_t o = w32_place(s, w32_thr(tau));
    uint32_t w[5];
#pragma unroll
    for (int b = 0; b < 5; ++b) w[b] = w32_place(s, w32_reg(1 << b));
    auto entry = [&](int i) -> uint32_t {
        uint32_t oi = o;
#pragma unroll
        for (int b = 0; b < 5; ++b)
            if (i & (1 << b)) oi += w[b];
        return oi;
    };
    c64_t a[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) a[i] = Cx<float>::from(__ldg(reinterpret_cast<const float2 *>(s.own + entry(i))));
#pragma unroll
    for (int i = 0; i < 32; i += 4) tmem_put4(tmem + 2 * i, a + i);
#pragma unroll
    for (int i = 0; i < 32; ++i)
        a[i] = Cx<float>::from(__ldg(reinterpret_cast<const float2 *>(s.par + (entry(i) ^ s.xo))));
#pragma unroll
    for (int i = 0; i < 32; i += 4) tmem_put4(tmem + 64 + 2 * i, a + i);
    tc_wait_st();
}

// Products of the filled factors for the shift whose register-index bits
// differ from the filled one's by 4 * d (d < 8): conj(partner[i ^ 4 d]) own[i].
__device__ __forceinline__ void w32_products(c64_t (&v)[32], uint32_t tmem, uint32_t d) {
    uint32_t a[2][8], b[2][8];
    tmem_ld8(tmem, a[0]);
    tmem_ld8(tmem + 64 + (d << 3), b[0]);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        tmem_wait_ld(a[i & 1], b[i & 1]);
        if (i < 7) {
            tmem_ld8(tmem + 8 * (i + 1), a[(i + 1) & 1]);
            tmem_ld8(tmem + 64 + (((uint32_t)(i + 1) ^ d) << 3), b[(i + 1) & 1]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            v[4 * i + q] = conj_mul<float>(__uint_as_float(b[i & 1][2 * q]), __uint_as_float(b[i & 1][2 * q + 1]),
                                           __uint_as_float(a[i & 1][2 * q]), __uint_as_float(a[i & 1][2 * q + 1]));
    }
}

// ----------------------------------------------------------------- powers

// acc + the 2 alpha-th powers of the real and imaginary parts of x, in FP32;
// A = alpha, or 0 for an order known at run time only, -1 for one of 2 x.
template <int A>
__device__ __forceinline__ c64_t w32_acc(c64_t acc, c64_t x, int alpha) {
    if constexpr (A < 0) x = Cx<float>::add(x, x);
    const c64_t sq = Cx<float>::mul(x, x);
    if constexpr (A == 2) return Cx<float>::fma(sq, sq, acc);
    c64_t p = sq;
    if constexpr (A > 2) {
#pragma unroll
        for (int k = 1; k < A; ++k) p = Cx<float>::mul(p, sq);
    } else {
        for (int k = 1; k < alpha; ++k) p = Cx<float>::mul(p, sq);
    }
    return Cx<float>::add(acc, p);
}

__device__ __forceinline__ double w32_flush(c64_t acc) {
    float a, b;
    Cx<float>::unpack(acc, a, b);
    return (double)(a + b);
}

// The thread's sum over its 32 packed values: FP32 over 16, FP64 above.
template <int A>
__device__ __forceinline__ double w32_pow_a(const c64_t (&v)[32], int alpha) {
    c64_t p = Cx<float>::zero(), q = Cx<float>::zero();
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        p = w32_acc<A>(p, v[i], alpha);
        q = w32_acc<A>(q, v[16 + i], alpha);
    }
    return w32_flush(p) + w32_flush(q);
}

__device__ __forceinline__ double w32_pow(const c64_t (&v)[32], int alpha) {
    switch (alpha) {
        case 2: return w32_pow_a<2>(v, alpha);
        case 3: return w32_pow_a<3>(v, alpha);
        case 4: return w32_pow_a<4>(v, alpha);
        default: return w32_pow_a<0>(v, alpha);
    }
}

__device__ __forceinline__ double warp_sum(double s) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    return s;
}

}  // namespace dev
}  // namespace sre
