// sre_tile.cuh -- in-CTA Walsh-Hadamard machinery on a tile of 2^12 complex
// entries held by 256 threads (16 entries each, i.e. 4 "register bits").
//
// The transform is the unnormalised WHT of the supplement's FWHT section:
// stage b maps each pair (a, c) of entries whose indices differ only in bit b
// to (a + c, a - c).  Stages commute, so the 12 bits are done in three rounds
// of four: a round does the butterflies over four index bits entirely in
// registers; between rounds the tile is rewritten through shared memory so
// that the next four bits become the register bits.
//
// Round layouts (tid in [0, 256), register slot i in [0, 16)):
//   round 0: e = tid << 4 | i                          (bits 0-3 in registers)
//   round 1: e = (tid >> 4) << 8 | i << 4 | (tid & 15)  (bits 4-7)
//   round 2: e = i << 8 | tid                          (bits 8-11)
// Shared memory stores entry e at pad(e) = e + (e >> 4): one spare slot per
// 16 entries.  Every round's stores and loads, and the XOR-shifted partner
// reads of the single-tile kernel, then hit distinct banks for 8- and
// 16-byte elements, and the address of slot i is the thread's base plus a
// compile-time offset.
//
// FP32 complex values live in one 64-bit register pair and are combined with
// the packed add/sub/mul/fma.rn.f32x2 instructions of sm_100+ (two IEEE
// round-to-nearest FP32 operations per instruction: the same results as
// scalar FP32 at half the instruction count).
//
// The FP64 mode transforms 64-bit fixed point (struct fx): an FP64 product is
// rounded to a multiple of 2^(k - 63) and every butterfly is an exact integer
// addition.  2^k bounds the values that the next four bits make, so nothing
// overflows; the unit follows their growth, rounded every four bits.  The bounds
// come from the tile's products themselves: the largest one, times 16 and 256,
// and the sums of their absolute parts, which no partial sum exceeds.  (Bounds
// from the norms of the factors are far too wide where their large entries do
// not meet: for a state close to a basis state a shift of high weight lost all
// its digits.)  Above the tile each block carries its own unit and bound into
// the transform over the blocks (FxExp).  Per-shift sums against 80-bit
// arithmetic, N = 6..16, Haar, product, near-basis, stabilizer and decaying
// states: at most 7e-16 off, as with FP64 butterflies.  The reason for fixed
// point is the pipe: GB300 runs 2 FP64 operations per clock and SM, against some
// 40 64-bit integer additions.  FP64 operations are left for the product (4 per
// entry) and the powers (4 per entry); both conversions are integer code, since
// F2I and I2F run at the FP64 rate too, and so are the bounds.  Measured: all
// shifts of an N = 16 state 47.5 ms (FP64 butterflies, full transforms below x =
// 4096: 178 ms; units from the factors' norms, known before the products: 46.0
// ms), 60 states of N = 12 11.3 ms with their evolution (61.9 ms; 10.5 ms); the
// FP64 pipe is busy 62 to 71 % of the time, and waits while the products of a
// tile are converted.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace sre {
namespace dev {

template <typename R> struct V2;
template <> struct V2<float> { using T = float2; };
template <> struct V2<double> { using T = double2; };
struct fx {};  // FP64 state, fixed-point transform
template <> struct V2<fx> { using T = double2; };
template <typename R> struct Real { using T = R; };
template <> struct Real<fx> { using T = double; };
template <typename R> using real_t = typename Real<R>::T;  // partial sums within a thread
template <typename R> using v2_t = typename V2<R>::T;

constexpr int kTileSlots = 4096 + 256;  // padded shared-memory tile
__host__ __device__ constexpr int pad(int e) { return e + (e >> 4); }

// ------------------------------------------------------------ complex ops
template <typename R> struct Cx;

template <> struct Cx<float> {
    using T = unsigned long long;  // (re, im) packed: re in the low half
    static __device__ __forceinline__ T pack(float re, float im) {
        T d;
        asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(re), "f"(im));
        return d;
    }
    static __device__ __forceinline__ void unpack(T v, float &re, float &im) {
        asm("mov.b64 {%0, %1}, %2;" : "=f"(re), "=f"(im) : "l"(v));
    }
    static __device__ __forceinline__ T add(T a, T b) {
        T d;
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
        return d;
    }
    static __device__ __forceinline__ T sub(T a, T b) {
        T d;
        asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
        return d;
    }
    static __device__ __forceinline__ T mul(T a, T b) {
        T d;
        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
        return d;
    }
    static __device__ __forceinline__ T fma(T a, T b, T c) {
        T d;
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
        return d;
    }
    static __device__ __forceinline__ T zero() { return 0ull; }
    static __device__ __forceinline__ T from(float2 v) { return pack(v.x, v.y); }
    static __device__ __forceinline__ float2 to(T v) {
        float2 r;
        unpack(v, r.x, r.y);
        return r;
    }
};

template <> struct Cx<fx> {
    using T = longlong2;
    static __device__ __forceinline__ T add(T a, T b) { return make_longlong2(a.x + b.x, a.y + b.y); }
    static __device__ __forceinline__ T sub(T a, T b) { return make_longlong2(a.x - b.x, a.y - b.y); }
    static __device__ __forceinline__ T zero() { return make_longlong2(0, 0); }
    static __device__ __forceinline__ T from(double2 v) {
        return make_longlong2(__double_as_longlong(v.x), __double_as_longlong(v.y));
    }
    static __device__ __forceinline__ double2 to(T v) {
        return make_double2(__longlong_as_double(v.x), __longlong_as_double(v.y));
    }
};

template <typename R> using cx_t = typename Cx<R>::T;

// conj(b) * a for scalar factors, packed.
template <typename R>
__device__ __forceinline__ cx_t<R> conj_mul(R br, R bi, R ar, R ai) {
    return Cx<R>::pack(br * ar + bi * ai, br * ai - bi * ar);
}

// Marks a tile with a product that is not a finite number (exponents of finite
// ones lie within +-1100).
constexpr int kFxNonFinite = 0x7fff;

// From unit 2^(k1 - 63) to the coarser 2^(k2 - 63), q = k2 - k1, rounded half
// up: the last bit shifted out is added afterwards, since a + 2^(q - 1) leaves 64
// bits for a near full scale.
__host__ __device__ __forceinline__ long long fx_shift(long long a, int q) {
    if (q <= 0) return a;
    if (q > 62) return 0;
    const long long t = a >> (q - 1);
    return (t >> 1) + (t & 1);
}
// The same for 0 <= q <= 8 and |a| <= 2^63 - 2^10, which all partial sums of a
// tile keep (a product has 53 bits).
__host__ __device__ __forceinline__ long long fx_shift_few(long long a, int q) { return (a + ((1ll << q) >> 1)) >> q; }

// round(p 2^(63 - k)), |p| < 2^k; the magnitude's high word, `down` places down,
// is added to sum.  The mantissa, 10 bits up, moves right by what its exponent
// lacks to the top; half of the last place is added first.
__device__ __forceinline__ long long fx_from(double p, int k, int down, unsigned &sum) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(p);
    const int e = (int)(b >> 52) & 2047;
    // shift left by e - 1075 + 63 - k in all, 10 of them already done
    const int q = 1022 - e + k;
    const unsigned long long m =
        (((b & 0xfffffffffffffull) | (e ? 1ull << 52 : 0ull)) << 10) + ((1ull << (q & 63)) >> 1);
    const long long r = (unsigned)q < 64 ? (long long)(m >> (q & 63)) : 0;  // zero, or below half a unit
    sum += (unsigned)(r >> 32) >> down;
    return (long long)b < 0 ? -r : r;
}

// |a| 2^-63 as a double (the sign does not matter to even powers), rounded to
// 53 bits; a carry out of the mantissa moves on into the exponent.
__device__ __forceinline__ double fx_abs(long long a) {
    const unsigned long long u = (unsigned long long)(a < 0 ? -a : a);
    const int lz = __clzll((long long)u);
    const unsigned long long n = u << (lz & 63);
    const unsigned long long m = (n >> 11) + ((n >> 10) & 1) + ((unsigned long long)(1022 - lz) << 52);
    return u ? __longlong_as_double((long long)m) : 0.0;
}

// g_x(t) = conj(phi_{t^x}) phi_t from the factors b = phi_{t^x}, a = phi_t, or
// for x = 0 (ZERO) W's input ((g0 + g1) / 2, (g0 - g1) / 2) from the two halves
// of g_0.  fx: the bits of the FP64 values, which fx_tile converts.
template <typename R, bool ZERO>
__device__ __forceinline__ cx_t<R> pair_value(v2_t<R> b, v2_t<R> a) {
    using T = real_t<R>;
    T re, im;
    if constexpr (ZERO) {
        const T g0 = a.x * a.x + a.y * a.y, g1 = b.x * b.x + b.y * b.y;
        re = T(0.5) * (g0 + g1);
        im = T(0.5) * (g0 - g1);
    } else {
        re = b.x * a.x + b.y * a.y;
        im = b.x * a.y - b.y * a.x;
    }
    if constexpr (sizeof(cx_t<R>) == 8)
        return Cx<R>::pack(re, im);
    else
        return Cx<fx>::from(make_double2(re, im));
}

// FP32: shifts below 4096 run on doubled products, so that their transforms are
// A, not W = A / 2.  The doubling is exact; the powers of W leave the range of
// FP32 where those of A do not (order 14 at N = 12: all digits of a sum of
// shifts).  From 4096 up, where states have twice the entries and more, it is W.
__device__ __forceinline__ bool fp32_doubled(uint64_t x) { return x < 4096; }
// Factor of an FP32 sum of powers: 1 for A, 2^(2 alpha) for W.
__device__ __forceinline__ double fp32_scale(bool doubled, int alpha) {
    return doubled ? 1.0 : (double)(1ull << (2 * alpha));
}

// A sum of (Re W)^(2 alpha) + (Im W)^(2 alpha) over fixed-point values of unit
// exponent k, times 2^(2 alpha) for the halving and the unit 2^k to the same
// power (NaN for a state without a finite norm, whose fixed-point values mean
// nothing).  The power alone may leave the range of a double where its product
// with the sum does not.
__device__ __forceinline__ double fx_scale(double s, int alpha, int k) {
    if (k == kFxNonFinite) return __longlong_as_double(0x7ff8000000000000ll);
    return scalbn(s, 2 * alpha * (1 + k));
}

// Where one shift finds the factors of a 4096-entry block of t' (t with the
// pivot bit removed): own entry e at place(e) from `own`, its partner at
// place(e) ^ xo from `par`.
template <typename V>
struct BlockPair {
    const V *own, *par;
    int xo, pivot;  // pivot 12: it lies above the block
    bool zero;      // x = 0: the two halves of g_0
    __device__ __forceinline__ int place(int e) const {
        if (pivot == 12) return e;
        const int lo = e & ((1 << pivot) - 1);
        return ((e - lo) << 1) | lo;
    }
};

template <typename V>
__device__ __forceinline__ BlockPair<V> block_pair(const V *psi, int N, uint64_t x, int tp) {
    BlockPair<V> s;
    s.zero = x == 0;
    const uint64_t xe = s.zero ? 1ull << (N - 1) : x;
    const int j = 63 - __clzll((long long)xe);
    if (j >= 12) {
        const uint64_t th = (((uint64_t)tp >> (j - 12)) << (j - 11)) | ((uint64_t)tp & ((1ull << (j - 12)) - 1));
        s.own = psi + (th << 12);
        s.par = psi + ((th ^ (xe >> 12)) << 12);
        s.xo = (int)(xe & 4095);
        s.pivot = 12;
    } else {
        s.own = s.par = psi + ((uint64_t)tp << 13);
        s.xo = (int)xe;
        s.pivot = j;
    }
    return s;
}

template <int K> __device__ __forceinline__ int elem(int tid, int i);
template <> __device__ __forceinline__ int elem<0>(int tid, int i) { return (tid << 4) | i; }
template <> __device__ __forceinline__ int elem<1>(int tid, int i) {
    return ((tid >> 4) << 8) | (i << 4) | (tid & 15);
}
template <> __device__ __forceinline__ int elem<2>(int tid, int i) { return (i << 8) | tid; }

// Products of a block in round-2 layout (e = i << 8 | tid), any pivot; FP32 ones
// doubled where the pivot lies inside the block (fp32_doubled).
template <typename R, bool ZERO>
__device__ __forceinline__ void block_values_z(cx_t<R> (&v)[16], const BlockPair<v2_t<R>> &s, int tid) {
    const int o = s.place(tid), w0 = s.place(256), w1 = s.place(512), w2 = s.place(1024), w3 = s.place(2048);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int e = o + ((i & 1) ? w0 : 0) + ((i & 2) ? w1 : 0) + ((i & 4) ? w2 : 0) + ((i & 8) ? w3 : 0);
        v[i] = pair_value<R, ZERO>(__ldg(s.par + (e ^ s.xo)), __ldg(s.own + e));
        if constexpr (sizeof(cx_t<R>) == 8) v[i] = Cx<R>::add(v[i], v[i]);
    }
}

template <typename R>
__device__ __forceinline__ void block_values(cx_t<R> (&v)[16], const BlockPair<v2_t<R>> &s, int tid) {
    if (s.zero)
        block_values_z<R, true>(v, s, tid);
    else
        block_values_z<R, false>(v, s, tid);
}

// Butterflies over register bits j in [0, 4) whose tile bit 4K + j < NB.
template <int K, int NB, typename R>
__device__ __forceinline__ void reg_stages(cx_t<R> (&v)[16]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (4 * K + j < NB) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                if (!(i & (1 << j))) {
                    const int p = i | (1 << j);
                    const cx_t<R> a = v[i], b = v[p];
                    v[i] = Cx<R>::add(a, b);
                    v[p] = Cx<R>::sub(a, b);
                }
            }
        }
    }
}

// Move the tile from round-KA layout to round-KB layout through `buf`
// (kTileSlots entries).  Moves between rounds 0 and 1 exchange register bits
// with thread bits 0-3, i.e. data moves only inside groups of 16 threads of
// one warp and each warp touches only its own part of the buffer: they are
// ordered with __syncwarp (WARP = true).  Moves between rounds 1 and 2
// exchange with thread bits 4-7 (across warps) and need a CTA barrier; their
// buffer must not be the one the previous tile's cross-warp move read
// (callers alternate two buffers).
template <int KA, int KB, bool WARP, typename R>
__device__ __forceinline__ void relayout(cx_t<R> (&v)[16], v2_t<R> *buf, int tid) {
    if (WARP) __syncwarp();
#pragma unroll
    for (int i = 0; i < 16; ++i) buf[pad(elem<KA>(tid, i))] = Cx<R>::to(v[i]);
    if (WARP)
        __syncwarp();
    else
        __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = Cx<R>::from(buf[pad(elem<KB>(tid, i))]);
}

// Transform over tile bits [0, NB), 0 <= NB <= 12, bits 0-3 first.  Input in
// round-0 layout; output in round-(max(NB-1,0)/4) layout.  bufA serves the
// warp-local round 0 -> 1 move (consecutive calls may share it); bufB the
// CTA-wide round 1 -> 2 move (NB > 8): consecutive calls must alternate bufB
// between two buffers.
template <int NB, typename R>
__device__ __forceinline__ void tile_fwht(cx_t<R> (&v)[16], v2_t<R> *bufA, v2_t<R> *bufB,
                                          int tid) {
    static_assert(NB >= 0 && NB <= 12, "tile transform covers 0..12 bits");
    reg_stages<0, NB, R>(v);
    if constexpr (NB > 4) {
        relayout<0, 1, true, R>(v, bufA, tid);
        reg_stages<1, NB, R>(v);
    }
    if constexpr (NB > 8) {
        relayout<1, 2, false, R>(v, bufB, tid);
        reg_stages<2, NB, R>(v);
    }
}

// Shared words of a CTA's fixed-point tile, per warp: exponent field of the
// largest product, sums of the absolute real and imaginary parts.
struct __align__(16) FxShared {
    int e[8];
    uint2 sums[8];
};

// A transformed tile: values are multiples of 2^(c - 63) below 2^c, and no sum
// of +-products of the tile reaches 2^s.
struct FxExp {
    int c, s;
};

__device__ __forceinline__ void fx_rescale(cx_t<fx> (&v)[16], int q) {
    if (q <= 0) return;
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = make_longlong2(fx_shift_few(v[i].x, q), fx_shift_few(v[i].y, q));
}

// 12-bit transform of the fixed-point mode, bits 8-11 first, of which the bits
// below NB are transformed: products (the bits of FP64 values) in round-2 layout
// in, round-0 layout out.  The first group of stages runs in units of each
// warp's own, so that the bounds of the tile meet at the barrier of the
// CTA-wide move: after it register i holds what warp i / 2 wrote.  One buffer
// serves both moves (after the CTA-wide one each warp stays in its own part of
// it); the barrier before it keeps the previous tile's readers ahead.
template <int NB>
__device__ __forceinline__ FxExp fx_tile(cx_t<fx> (&v)[16], double2 *buf, int tid, FxShared &sh) {
    // stages of each group
    constexpr int GA = NB > 8 ? NB - 8 : 0, GB = NB > 8 ? 4 : NB > 4 ? NB - 4 : 0, GC = NB > 4 ? 4 : NB;
    const int lane = tid & 31, warp = tid >> 5;
    unsigned m = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i)
        m = max(m, max((unsigned)(v[i].x >> 32) & 0x7fffffffu, (unsigned)(v[i].y >> 32) & 0x7fffffffu));
    const int e = (int)(__reduce_max_sync(0xffffffffu, m) >> 20);  // the warp's products: below 2^(e - 1022)
    // sums of |re| and |im|, each entry rounded up to 2^(e - 1022 - 27): 16
    // entries make 2^31 + 16 at most, then 2^(e - 1022 - 22) for the warp
    unsigned sr = 16, si = 16;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        v[i].x = fx_from(__longlong_as_double(v[i].x), e - 1022 + GA, 4 - GA, sr);
        v[i].y = fx_from(__longlong_as_double(v[i].y), e - 1022 + GA, 4 - GA, si);
    }
    sr = __reduce_add_sync(0xffffffffu, (sr >> 5) + 1);
    si = __reduce_add_sync(0xffffffffu, (si >> 5) + 1);
    reg_stages<2, NB, fx>(v);
    __syncthreads();
    if (lane == 0) {
        sh.e[warp] = e;
        sh.sums[warp] = make_uint2(sr, si);
    }
    relayout<2, 1, false, fx>(v, buf, tid);
    // the tile's largest exponent, and its sums in units of 2^(most - 1022 - 19),
    // with one unit more: the rescaling below moves a sum by less (2^8 units
    // of the coarsest, 2^(c - 63))
    const int ew = sh.e[lane & 7], most = __reduce_max_sync(0xffffffffu, ew);
    const uint2 t = sh.sums[lane & 7];
    const int d = min(most - ew + 3, 31);
    sr = __reduce_add_sync(0xffffffffu, lane < 8 ? (t.x >> d) + 1 : 0) + 1;
    si = __reduce_add_sync(0xffffffffu, lane < 8 ? (t.y >> d) + 1 : 0) + 1;
    FxExp u;
    u.s = most - 1022 - 19 + 32 - __clz(max(sr, si));
    const int ka = most - 1022 + GA, kb = min(max(u.s, ka), ka + GB);
    u.c = min(max(u.s, kb), kb + GC);
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        const int q = kb - (sh.e[w] - 1022 + GA);
        if (q > 8) {
#pragma unroll
            for (int i = 2 * w; i < 2 * w + 2; ++i) v[i] = make_longlong2(fx_shift(v[i].x, q), fx_shift(v[i].y, q));
        } else if (q > 0) {
#pragma unroll
            for (int i = 2 * w; i < 2 * w + 2; ++i)
                v[i] = make_longlong2(fx_shift_few(v[i].x, q), fx_shift_few(v[i].y, q));
        }
    }
    reg_stages<1, NB, fx>(v);
    fx_rescale(v, u.c - kb);
    relayout<1, 0, true, fx>(v, buf, tid);
    reg_stages<0, NB, fx>(v);
    if (most == 2047) u.c = u.s = kFxNonFinite;
    return u;
}

// Units of the transform over a shift's 2^H2 blocks: k[0] for its first four
// bits, k[1] and k[2] for the next ones; the last also for its results.  low: the
// smallest of the blocks' own.
template <int H2>
struct FxUnits {
    static constexpr int G0 = H2 < 4 ? H2 : 4, G1 = H2 < 4 ? 0 : H2 < 8 ? H2 - 4 : 4, G2 = H2 < 8 ? 0 : H2 - 8;
    int k[3], low;
};

// From the smallest and largest unit of the blocks and a bound 2^s of their sum.
template <int H2>
__device__ __forceinline__ FxUnits<H2> fx_units(int low, int cm, int s) {
    using U = FxUnits<H2>;
    U u;
    u.low = low;
    u.k[0] = min(max(s, cm), cm + U::G0);
    u.k[1] = min(max(s, u.k[0]), u.k[0] + U::G1);
    u.k[2] = min(max(s, u.k[1]), u.k[1] + U::G2);
    if (cm == kFxNonFinite) u.k[2] = kFxNonFinite;
    return u;
}

// The same from the blocks' exponents in global memory, by a warp.  Bounds are
// added as multiples of 2^(largest - 20), rounded up: 2^11 blocks fit 32 bits.
template <int H2>
__device__ __forceinline__ FxUnits<H2> fx_units(const short *c, const short *s) {
    constexpr int n = 1 << H2;
    const int lane = threadIdx.x & 31;
    int low = kFxNonFinite, cm = -0x8000, sm = -0x8000;
#pragma unroll 1
    for (int t = lane; t < n; t += 32) {
        const int ct = __ldcg(c + t);
        low = min(low, ct);
        cm = max(cm, ct);
        sm = max(sm, (int)__ldcg(s + t));
    }
    low = __reduce_min_sync(0xffffffffu, low);
    cm = __reduce_max_sync(0xffffffffu, cm);
    sm = __reduce_max_sync(0xffffffffu, sm);
    unsigned sum = 0;
#pragma unroll 1
    for (int t = lane; t < n; t += 32) sum += (1u << 20) >> min(sm - (int)__ldcg(s + t), 20);
    sum = __reduce_add_sync(0xffffffffu, sum);
    return fx_units<H2>(low, cm, sm - 20 + 32 - __clz(sum - 1));
}

// This thread's entries (round-0 layout, block = entry index mod 2^H2) from
// their blocks' units, c, to the unit k.
template <int H2>
struct FxAlign {
    static constexpr int n = H2 < 4 ? 1 << H2 : 16;
    __align__(16) short q[n];
    __device__ __forceinline__ FxAlign(const short *c, int tid) {
        const short *p = c + ((tid << 4) & ((1 << H2) - 1));
        if constexpr (n == 4) {
            *reinterpret_cast<int2 *>(q) = __ldcg(reinterpret_cast<const int2 *>(p));
        } else {
#pragma unroll
            for (int j = 0; j < n; j += 8)
                *reinterpret_cast<int4 *>(q + j) = __ldcg(reinterpret_cast<const int4 *>(p + j));
        }
    }
    __device__ __forceinline__ void operator()(cx_t<fx> (&v)[16], const FxUnits<H2> &u) const {
        const int k = u.k[0];
        // all but strongly decaying states (below four bits the units are uniform,
        // and two paths only cost registers)
        if (H2 >= 4 && k - u.low <= 8) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int d = k - q[i & (n - 1)];
                v[i] = make_longlong2(fx_shift_few(v[i].x, d), fx_shift_few(v[i].y, d));
            }
            return;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int d = k - q[i & (n - 1)];
            v[i] = make_longlong2(fx_shift(v[i].x, d), fx_shift(v[i].y, d));
        }
    }
};

// Transform over the 2^H2 blocks, round-0 layout in, units u.
template <int H2>
__device__ __forceinline__ void fx_rows(cx_t<fx> (&v)[16], double2 *buf, int tid, const FxUnits<H2> &u) {
    reg_stages<0, H2, fx>(v);
    if constexpr (H2 > 4) {
        fx_rescale(v, u.k[1] - u.k[0]);
        relayout<0, 1, true, fx>(v, buf, tid);
        reg_stages<1, H2, fx>(v);
    }
    if constexpr (H2 > 8) {
        fx_rescale(v, u.k[2] - u.k[1]);
        relayout<1, 2, false, fx>(v, buf, tid);
        reg_stages<2, H2, fx>(v);
    }
}

// Full 12-bit transform, bits 8-11 first: input in round-2 layout (thread
// tid holds e = i << 8 | tid, so loads of consecutive threads are
// contiguous), output in round-0 layout.  One CTA-wide move (bufB, to be
// alternated between consecutive calls) and one warp-local move (bufA).
template <typename R>
__device__ __forceinline__ void tile_fwht12_rev(cx_t<R> (&v)[16], v2_t<R> *bufA, v2_t<R> *bufB,
                                                int tid) {
    reg_stages<2, 12, R>(v);
    relayout<2, 1, false, R>(v, bufB, tid);
    reg_stages<1, 12, R>(v);
    relayout<1, 0, true, R>(v, bufA, tid);
    reg_stages<0, 12, R>(v);
}

// sum_i (Re F_i)^(2 A) + (Im F_i)^(2 A) over the thread's 16 entries, in FP32
// or FP64 (fx, in units of 2^k); A = 0: the order alpha known at run time only.
template <typename R, int A>
__device__ __forceinline__ real_t<R> sum_re_im_pow(const cx_t<R> (&v)[16], int alpha) {
    if constexpr (sizeof(cx_t<R>) == 8) {
        cx_t<R> acc = Cx<R>::zero();
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const cx_t<R> sq = Cx<R>::mul(v[i], v[i]);
            if constexpr (A == 2) {
                acc = Cx<R>::fma(sq, sq, acc);
                continue;
            }
            cx_t<R> p = sq;
            if constexpr (A > 0) {
#pragma unroll
                for (int k = 1; k < A; ++k) p = Cx<R>::mul(p, sq);
            } else {
                for (int k = 1; k < alpha; ++k) p = Cx<R>::mul(p, sq);
            }
            acc = Cx<R>::add(acc, p);
        }
        float a, b;
        Cx<R>::unpack(acc, a, b);
        return a + b;
    } else {
        double acc = 0.0, acd = 0.0;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const double re = fx_abs(v[i].x), im = fx_abs(v[i].y);
            const double s = re * re, t = im * im;
            double p = s, q = t;
            for (int k = 2; k < (A ? A : alpha); ++k) {
                p *= s;
                q *= t;
            }
            acc = __fma_rn(p, s, acc);
            acd = __fma_rn(q, t, acd);
        }
        return acc + acd;
    }
}

// The thread's share of the order-alpha sum of the halved form.
template <typename R>
__device__ __forceinline__ real_t<R> sum_order(const cx_t<R> (&v)[16], int alpha) {
    switch (alpha) {
        case 2: return sum_re_im_pow<R, 2>(v, alpha);
        case 3: return sum_re_im_pow<R, 3>(v, alpha);
        case 4: return sum_re_im_pow<R, 4>(v, alpha);
        default: return sum_re_im_pow<R, 0>(v, alpha);
    }
}

// Deterministic block-wide FP64 sum (fixed tree); result valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double *red /* kThreads/32 */) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0) {
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    }
    return s;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Drop a 128-byte L2 line without writing it back (its contents become
// undefined).  Used on inter-pass scratch once every reader is done with it.
__device__ __forceinline__ void discard_l2_line(const void *p) {
    asm volatile("discard.global.L2 [%0], 128;" ::"l"(p) : "memory");
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

}  // namespace dev
}  // namespace sre
