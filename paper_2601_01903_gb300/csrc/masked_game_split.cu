// Masked-model value function in float64 and float32 with layer 2 on the
// tensor cores, by exact digit splitting (hidden widths up to 128, d >= 7).
//
// v_x(S) = f(z), z_i = x_i for i in S and a background value otherwise, f the
// GELU MLP d -> h1 -> h2 -> 1 (the value function of Section 2.1; the
// interventional one of Section 4.1 averages f over the background rows).
// On the CUDA cores the h1 x h2 products of a coalition bound this function
// (float64: 0.5 multiply-adds per clock and lane quarter), and the float64
// GELUs come next.  Here
//
//   layer 2 is a product of integers: the activations of a tile and W2 are cut
//     to fixed point and written as balanced base-256 digits (float64: 7 digits =
//     56 bits, float32: 4 = 32 bits), each an exact FP16 number.  A product of two
//     digit matrices over K <= 128 has sums below 2^21, so all products of one
//     diagonal i + j = const add up exactly in one FP32 accumulator (at most 7 of
//     them, below 2^24): the Ozaki splitting (Ozaki, Ogita, Oishi & Rump,
//     "Error-free transformations of matrix multiplication", 2012) with fixed
//     digits.  Diagonals 0 .. 7 (float64, 34 products) or 0 .. 3 (float32, 10) are
//     kept: what is dropped is below the rounding of the last digit.  The
//     diagonals are put together in 64-bit integers (float64) or by three fused
//     multiply-adds (float32).
//   float64 everywhere else is 64-bit fixed point on the integer pipes, which
//     are some 60 times as wide as the float64 pipe of this part: layer-1
//     pre-activations are sums of integers (exact, by subset sums), GELU is
//     max(z, 0) - |z| Phi(-|z|) with the second term from a table of quintic
//     polynomials, layer 3 exact 32 x 32-bit products.
//
// Scales (all powers of two, so that none of them rounds anything):
//   a unit of layer 1 has an exponent E, from a bound of its pre-activations over
//     the instance's coalitions; its activations count in units of 2^E and its
//     column of W2 is multiplied by 2^E;
//   a row of W2 (so scaled) has an exponent of its own, undone where the
//     accumulators are drained, and in float64 a unit of layer 2 a format of its
//     own (62 bits from its bound down), undone in W3;
//   a coalition has an exponent e <= 0, from what its features and b1 can give any
//     unit, undone with the row's: coalitions of small features keep their digits.
// The model's own exponents, for features of size 2, serve the instances whose
// bounds they hold, so that one set of W2's slices serves many; an instance
// beyond them gets its own.
// The fixed point is taken where what it adds stays below the rounding of the
// type's own arithmetic:
//   the digits of a row of W2 end 2^-57 (2^-33) below its largest entry, a double
//     (float) loses 2^-54 (2^-25) of each product and about sqrt(terms) times that
//     in their sum: the largest entry may be up to EVEN max(12, 3 sqrt(terms)) times
//     the mean of the others', weighted by their bounds and averaged over the rows
//     by |W3|;
//   the GELU table is off by 2^-59 whatever the result, so in float64 no unit of
//     layer 2 may carry most of W3 (mu >= 8), W3 has to be even in the same sense
//     as W2, and a coalition may lie 2^-6 at most below the largest (row_span: less
//     for units of small pre-activations or an uneven W3); float32's pre-
//     activations go through floats, and its coalitions may lie 2^-34 below;
//   one feature may leave the others 2^-8 (float64) or 2^-34 of a unit's bound.
// A unit that no coalition can lift to -9 is left out (its GELU is 0).  Coalitions
// below row_span (slow_rows), and instances that the rules refuse, among them all
// with non-finite values (slow_tiles), are evaluated in the arithmetic of the type.
// (One exponent for all units of a layer, as this path had at first, lost the bits
// by which a unit, a bias or a coalition was smaller than the largest: 5e-2 of the
// values in float32 for one unit 2^28 above the others.)
//
// One CTA (16 warps) per SM walks a contiguous range of 128-coalition tiles:
// layer 1 of a tile into the digit slices in shared memory, one thread issues
// its MMAs, and while they run all warps do layers 2 (GELU) and 3 of the tile
// before, whose accumulators they drained into registers.
//
// Measured on one GB300: float64, 64 instances of a 14-64-64-1 model (2^20
// coalitions) 19.67 ms on masked_game_kernel, 0.80 ms here; float32, 8
// instances of a 16-128-128-1 model (2^19) 2.38 ms, 0.27 ms here.  Largest
// errors, coalition by coalition and against extended precision, are 0.3 to 0.9
// of masked_game_kernel's on even models and at most 1.7 times them over units,
// biases and features of other scales (2^-28 to 2^28, -1e8, 1e12).  An
// instance's scales take 1.7 us where the model's serve, 6 us where not, and the
// model's 6 us at the start.  Instances that are all refused take 0.4 to 0.5 of
// masked_game_kernel's time in float64; in float32 0.6 (128 x 128 units) to 1.2 (64 x
// 64, many tiles: 16 warps per SM hide less of the latencies than its 52), 0.4 to 0.5
// for few tiles.
// What bounds the fast path is the work of the GELUs at one CTA per SM (its
// accumulators take the tensor memory, its slices and table the shared memory).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#define TTFSI_GEMM_HELPERS_ONLY
#include "gemm_tcgen05.cuh"
#include "masked_game_split.h"
#include "tt_fsi.h"

namespace ttfsi_mgs {

using ttfsi_gemm::mbar_init;
using ttfsi_gemm::mbar_wait;
using ttfsi_gemm::mma_commit;
using ttfsi_gemm::smem_desc;
using ttfsi_gemm::smem_u32;

typedef long long i64;
typedef unsigned long long u64;

constexpr int ROWS = 128;              // coalitions per tile (MMA M)
constexpr int LOW = 7;                 // log2 ROWS
constexpr int KC = 64;                 // hidden units per K chunk (one 128-byte swizzled row)
constexpr int THREADS = 512;
constexpr int WARPS = THREADS / 32;
constexpr int MAXH = 128;
constexpr int SLICE_A = ROWS * 128;    // bytes of one digit slice of a chunk of activations

template <bool F64>
struct Cfg {
    static constexpr int NS = F64 ? 7 : 4;     // digits
    static constexpr int ND = F64 ? 8 : 4;     // diagonals = accumulators
    static constexpr int NW = F64 ? 64 : 128;  // layer-2 units per pass; ND * NW = 512 TMEM columns
    static constexpr int BITS = F64 ? 55 : 31; // fraction bits of the digit format
    static constexpr int CPT = NW / 4;         // accumulator columns per thread in the epilogue
    // what the fixed point serves (see above)
    static constexpr int EMIN = F64 ? 0 : -60, EMAX = F64 ? 19 : 60;  // exponents of a unit of layer 1
    static constexpr int SPAN = F64 ? 6 : 34;                         // bits between the largest row and a row
    static constexpr float LONE = F64 ? 0x1p-8f : 0x1p-34f;           // one feature against a unit's others
    static constexpr float TYPICAL = 2.f;                            // size of a feature that the model's scales allow for
    static constexpr float EVEN = F64 ? 1.5f : 4.f;                   // digits of W2 below the type's own
};

// ---- GELU in fixed point ---------------------------------------------------
// |z| Phi(-|z|) on intervals of width 2^-7, |z| < 8.75 (beyond it is below
// 2^-56 and taken as 0): per interval the quintic in tau = 256 (|z| - centre)
// that remains of its Taylor polynomial of degree 7 when the two highest
// Chebyshev terms are dropped, coefficients rounded to fixed point from the
// highest down: c0 (62 fraction bits), c1 (71), c2 (80; its low 16 bits hold
// c5), c3 (57), c4 (58), c5 (59).  Largest error against 160-bit arithmetic
// 2^-56.9, root mean square 2^-59.2 (float64's own rounding of a result near
// 1/3 is up to 2^-55).  The first row's c0 is 7 units lower than so rounded: the
// integer arithmetic then gives 0 at z = 0, and a model without biases exactly b3
// where all features are 0.
constexpr int TAB_INTERVALS = 1120;
constexpr int TAB_ROWS = TAB_INTERVALS + 1;
__device__ const ulonglong2 g_gelu_table[TAB_ROWS][2] = {
#include "gelu_table.inc"
};

// Pieces of 64-bit arithmetic on 32-bit words, shifts by less than 32 (the
// compiler's own 64-bit shifts by a variable also serve 32 and more).
__device__ __forceinline__ int hi32(i64 v) { return (int)(v >> 32); }
__device__ __forceinline__ unsigned lo32(i64 v) { return (unsigned)v; }
__device__ __forceinline__ i64 join(unsigned lo, int hi) { return ((i64)hi << 32) | lo; }
__device__ __forceinline__ i64 mad_wide(int a, int b, i64 c) {
    i64 r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
__device__ __forceinline__ i64 mul_wide(int a, int b) {
    i64 r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ i64 shr(i64 v, int k) {
    return join(__funnelshift_r(lo32(v), (unsigned)hi32(v), k), hi32(v) >> k);
}

// c + a b / 2^64 to within three units, on the multiply-add pipe alone (the
// product of the low halves is dropped; a_half is the low word of a over 2).
__device__ __forceinline__ i64 mul_hi_add(int a_hi, int a_half, i64 b, i64 c, int two) {
    const int mid = hi32(mad_wide(a_half, hi32(b), mul_wide(a_hi, (int)(lo32(b) >> 1))));
    return mad_wide(a_hi, hi32(b), mad_wide(mid, two, c));
}

// GELU of z = Z 2^(s - 62) as an integer of the same format, 0 <= s <= 19.  What
// bounds it is the integer ALU (half the issue rate), so shifts and adds are
// left to multiplications where the formats allow it.
__device__ __forceinline__ i64 gelu_fixed(i64 Z, int s, const ulonglong2 *tab, int two) {
    const int sign = hi32(Z) >> 31;
    const i64 m = (Z ^ join((unsigned)sign, sign)) - (i64)sign;
    const unsigned mh = (unsigned)hi32(m);
    const unsigned idx = min(mh >> (23 - s), (unsigned)TAB_INTERVALS);
    // tau 2^63: the bits below the index, about the centre
    const int t = (int)(__funnelshift_l(lo32(m), mh, 9 + s) ^ 0x80000000u);
    const unsigned tlow = lo32(m) << (9 + s);
    const ulonglong2 r0 = tab[2 * idx], r1 = tab[2 * idx + 1];
    const int u4 = (int)(r1.y >> 32) + __mulhi(t, (int)(short)(r1.x & 0xffff));
    const int u3 = (int)(unsigned)r1.y + __mulhi(t, u4);
    const int th = t >> 8, tl = (int)(__funnelshift_r(tlow, (unsigned)t, 8) >> 1);  // tau 2^55
    const i64 u2 = mad_wide(th, u3, mad_wide(__mulhi(tl, u3), two, (i64)r1.x));
    const i64 u1 = mul_hi_add(th, tl, u2, (i64)r0.y, two);
    const i64 h = mul_hi_add(th, tl, u1, (i64)r0.x, two);  // near z = 0 possibly a unit below 0
    return (Z & ~join((unsigned)sign, sign)) - shr(h, s);
}

// GELU in float32 without branches: max(z, 0) - t Phi(-t), t = |z|, with
// exp(t^2 / 2) Phi(-t) as a polynomial in s = 1 / (1 + 0.28 t) (weighted
// least squares over 0 <= t <= 6.5, refitted to an even error; that of the
// product is 3.4e-9, below the rounding of float32).
__device__ __forceinline__ float gelu_fast(float z) {
    const float t = fabsf(z);
    float s, e;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(fmaf(0.28f, t, 1.0f)));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(t * t * -0.72134752044448170f));
    float p = fmaf(-0.10755508235538286f, s, 0.39699074731224754f);
    p = fmaf(p, s, -0.24851913789490362f);
    p = fmaf(p, s, 0.27818327722545133f);
    p = fmaf(p, s, 0.06379108976018237f);
    p = fmaf(p, s, 0.11710905724886507f);
    return fmaf(-(t * s) * e, p, fmaxf(z, 0.f));
}
__device__ __forceinline__ float gelu_of(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752440f)); }
__device__ __forceinline__ double gelu_of(double z) { return 0.5 * z * (1.0 + erf(z * 0.70710678118654752440)); }

// ---- small helpers ------------------------------------------------------------
// v 2^f rounded to an integer (float64 bits to integer, no float64 arithmetic);
// the caller keeps |v| 2^f below 2^62.
__device__ __forceinline__ i64 fix(double v, int f) {
    const u64 b = (u64)__double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0) return 0;
    const u64 mant = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = f + e - 1075;
    u64 r;
    if (sh >= 0)
        r = sh < 64 ? mant << sh : 0;
    else
        r = sh > -64 ? (mant + (1ull << (-sh - 1))) >> -sh : 0;
    return (b >> 63) ? -(i64)r : (i64)r;
}

// An exponent c with v < 2^c (v >= 0; -127 for 0, 129 for infinities and NaN).
__device__ __forceinline__ int exp_above(float v) {
    const int e = (int)((__float_as_uint(v) >> 23) & 0xff);
    return e == 0 ? -127 : e - 126;
}

// |v| cut to a float without float64 arithmetic: 0 below 2^-126, infinite from
// 2^127 on and for NaN.
__device__ __forceinline__ float magnitude(double v) {
    const u64 b = (u64)__double_as_longlong(v);
    const unsigned hi = (unsigned)(b >> 32) & 0x7fffffffu, e = hi >> 20;
    const unsigned f = ((e - 896) << 23) | ((hi & 0xfffffu) << 3) | ((unsigned)b >> 29);
    return __uint_as_float(e < 1023 - 126 ? 0u : e > 1023 + 126 ? 0x7f800000u : f);
}

// 2^e as a float, -126 <= e <= 127.
__device__ __forceinline__ float pow2(int e) { return __uint_as_float((unsigned)(e + 127) << 23); }

// Writes the digits of two neighbouring K elements to the slices.  The values
// come biased, so that each byte holds its digit + 128; the FP16 pattern
// 0x64 byte is 1024 + byte, and 1152 less is the digit.
__device__ __forceinline__ unsigned prmt(unsigned a, unsigned b, unsigned sel) { return __byte_perm(a, b, sel); }
__device__ __forceinline__ void put_pair(unsigned char *dst, unsigned two) {
    unsigned r;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(two), "r"(0x64806480u));
    *reinterpret_cast<unsigned *>(dst) = r;
}
// four digits of a word each, most significant first
__device__ __forceinline__ void put_four(unsigned char *dst, int slice_bytes, unsigned a, unsigned b) {
    const unsigned hi = prmt(a, b, 0x7632), lo = prmt(a, b, 0x5410);  // bytes 2, 3 and 0, 1 of both
    put_pair(dst, prmt(hi, 0x64646464u, 0x4341));
    put_pair(dst + slice_bytes, prmt(hi, 0x64646464u, 0x4240));
    put_pair(dst + 2 * slice_bytes, prmt(lo, 0x64646464u, 0x4341));
    put_pair(dst + 3 * slice_bytes, prmt(lo, 0x64646464u, 0x4240));
}
constexpr u64 BIAS7 = 0x0080808080808080ull;  // + 128 in each of seven bytes
constexpr unsigned BIAS4 = 0x80808080u;
// float64: values + BIAS7 (below 2^56)
__device__ __forceinline__ void put_digits(unsigned char *dst, int slice_bytes, u64 a, u64 b) {
    const unsigned ah = (unsigned)(a >> 32) | 0x64000000u, bh = (unsigned)(b >> 32) | 0x64000000u;
    put_pair(dst, prmt(ah, bh, 0x7632));
    put_pair(dst + slice_bytes, prmt(ah, bh, 0x7531));
    put_pair(dst + 2 * slice_bytes, prmt(ah, bh, 0x7430));
    put_four(dst + 3 * slice_bytes, slice_bytes, (unsigned)a, (unsigned)b);
}
// float32: values + BIAS4
__device__ __forceinline__ void put_digits(unsigned char *dst, int slice_bytes, unsigned a, unsigned b) {
    put_four(dst, slice_bytes, a, b);
}

// Byte offset of the K pair u (elements 2u, 2u + 1) of row r in a 128-byte
// swizzled slice.
__device__ __forceinline__ int pair_offset(int r, int u) { return r * 128 + (((u >> 2) ^ (r & 7)) << 4) + (u & 3) * 4; }

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void tmem_ld8(uint32_t addr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(addr));
}

struct Args {
    const double *W1, *b1, *W2, *b2, *W3;
    double b3;
    const float *W2f, *b2f, *W3f;  // float32 path
    const double *x, *bg;
    void *v;
    int n_bg, d, h1, h2;
    int halves;  // 1: two CTAs per tile, each for 64 of its coalitions
    long long n_tiles;
    double scale;
    // powers of two that the compiler must not see through: it would turn the
    // multiply-adds by them into shifts and adds on the busier integer ALU
    int two, unit[4];  // 2; 2^24, 2^16, 2^8, 1
};

// Shared memory (dynamic; the two operand regions on 1024-byte boundaries).
template <bool F64>
struct Smem {
    using C = Cfg<F64>;
    static constexpr int CHUNKS = F64 ? 1 : 2;  // K chunks whose tables and W2 slices are kept (float32: all)
    static constexpr int A = 0;
    static constexpr int W = A + C::NS * SLICE_A;
    static constexpr int TAB = W + CHUNKS * C::NS * C::NW * 128;
    static constexpr int PH = TAB + (F64 ? TAB_ROWS * 32 : 0);  // [16][KC] pre-activations by bits 3 .. 6
    static constexpr int DL = PH + 16 * KC * (F64 ? 8 : 4);     // [CHUNKS][7][KC] i64: a low feature joins
    static constexpr int DF = DL + CHUNKS * LOW * KC * 8;       // float32: [CHUNKS][3][KC], the first three as floats
    static constexpr int PART = DF + (F64 ? 0 : CHUNKS * 3 * KC * 4);  // [3][ROWS] row sums of column groups 1 .. 3
    static constexpr int COL = PART + 3 * ROWS * (F64 ? 16 : 4);  // [NW] 16 bytes: b2 and W3 in fixed point | b2, W3, 2^ew
    static constexpr int CS = COL + C::NW * 16;                 // float64: [NW] 62 - f
    static constexpr int CE = CS + (F64 ? C::NW * 4 : 0);       // float64: [NW] ew + f - 38
    static constexpr int SE = CE + (F64 ? C::NW * 4 : 0);       // [MAXH] exponent of a unit of layer 1 + 64, kDead
    static constexpr int EW = SE + MAXH * 4;                    // [MAXH] exponent of a row of W2, or kDead
    static constexpr int FN = EW + MAXH * 4;                    // float64: [MAXH] fraction bits of a unit of layer 2
    static constexpr int ER = FN + (F64 ? MAXH * 4 : 0);        // [2][ROWS], double-buffered: the rows' exponents e, a byte each | 2^(31 - e), floats
    static constexpr int MW = ER + 2 * ROWS * (F64 ? 1 : 4);    // [32] float: a feature's largest scaled weight, b1's
    static constexpr int MB = MW + 32 * 4;                      // [32] float: a feature's largest background value
    static constexpr int MX = MB + 32 * 4;                      // [32] float2: what a feature gives a row, in it and not
    static constexpr int RL = MX + 32 * 8;                      // [ROWS] float: what the low features and b1 give a row
    static constexpr int END = RL + ROWS * 4;
    static constexpr int BYTES = END + 1024;
};
static_assert(Smem<true>::BYTES <= 232448 - 1024 && Smem<false>::BYTES <= 232448 - 1024, "fits one CTA per SM");
constexpr int kDead = 1 << 10;

// N values over the CTA, the first NSUM of them summed (in a fixed order), the
// rest maximised (none of them negative); every thread gets them.
template <int N, int NSUM>
__device__ __forceinline__ void block_reduce(float (&v)[N], float (&red)[WARPS][10]) {
    static_assert(N <= 10, "red");
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float u = __shfl_xor_sync(0xffffffffu, v[i], o);
            v[i] = i < NSUM ? v[i] + u : fmaxf(v[i], u);
        }
    __syncthreads();
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int i = 0; i < N; ++i) red[threadIdx.x >> 5][i] = v[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N; ++i) {
        v[i] = red[threadIdx.x & (WARPS - 1)][i];
#pragma unroll
        for (int o = WARPS / 2; o > 0; o >>= 1) {
            const float u = __shfl_xor_sync(0xffffffffu, v[i], o);
            v[i] = i < NSUM ? v[i] + u : fmaxf(v[i], u);
        }
    }
}

template <typename T>
struct Weights;
template <>
struct Weights<double> {
    static __device__ __forceinline__ const double *w2(const Args &a) { return a.W2; }
    static __device__ __forceinline__ const double *b2(const Args &a) { return a.b2; }
    static __device__ __forceinline__ const double *w3(const Args &a) { return a.W3; }
};
template <>
struct Weights<float> {
    static __device__ __forceinline__ const float *w2(const Args &a) { return a.W2f; }
    static __device__ __forceinline__ const float *b2(const Args &a) { return a.b2f; }
    static __device__ __forceinline__ const float *w3(const Args &a) { return a.W3f; }
};

// GELU of the rows below: erff, and in float64 (whose pipe bounds them) the table
// where its 2^-59 is below the rounding of the result: for 2^-4 <= |z| < 8, z
// an exact multiple of 2^-58; below, z Phi(z) = z / 2 + z^2 (1 - z^2 / 6 + z^4 / 40 -
// ...) / sqrt(2 pi), Taylor's series of Phi.
__device__ __forceinline__ float gelu_slow(float z, const ulonglong2 *, int) { return gelu_of(z); }
__device__ __forceinline__ double gelu_slow(double z, const ulonglong2 *tab, int two) {
    const float m = magnitude(z);
    if (m >= 0.0625f && m < 8.f) {
        const int s = m < 1.f ? 1 : 4;
        return (double)gelu_fixed(fix(z, 62 - s), s, tab, two) * (m < 1.f ? 0x1p-61 : 0x1p-58);
    }
    if (m < 0.0625f) {
        const double y = z * z;
        double p = fma(y, 1.0 / 599040, -1.0 / 42240);
        p = fma(y, p, 1.0 / 3456);
        p = fma(y, p, -1.0 / 336);
        p = fma(y, p, 1.0 / 40);
        p = fma(y, p, -1.0 / 6);
        p = fma(y, p, 1.0);
        return fma(y * 0.39894228040143267794, p, 0.5 * z);
    }
    if (m >= 8.75f && m < 1e38f) return z > 0.0 ? z : -0.0;  // (1 + erf is 2 or 0)
    return gelu_of(z);
}

// Layer 2 (GELU) and layer 3 of one coalition for units n0, n0 + step, ...,
// NB neighbours at a time.
template <typename T, int NB>
__device__ __forceinline__ T slow_units(const Args &a, const T *row, int n0, int step, const ulonglong2 *tab) {
    const T *w2 = Weights<T>::w2(a), *b2 = Weights<T>::b2(a), *w3 = Weights<T>::w3(a);
    const bool by_four = sizeof(T) == 4 && a.h1 % 4 == 0 && (reinterpret_cast<uintptr_t>(w2) & 15) == 0;
    T sum = 0;
    for (int n = n0; n < a.h2; n += step) {
        T acc[NB];
        const T *w[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const int m = min(n + k, a.h2 - 1);
            acc[k] = b2[m];
            w[k] = w2 + m * a.h1;
        }
        int i = 0;
        if constexpr (sizeof(T) == 4) {
            if (by_four) {
#pragma unroll 2
                for (; i < a.h1; i += 4) {
#pragma unroll
                    for (int k = 0; k < NB; ++k) {
                        const float4 v = __ldg(reinterpret_cast<const float4 *>(w[k] + i));
                        acc[k] += v.x * row[i];
                        acc[k] += v.y * row[i + 1];
                        acc[k] += v.z * row[i + 2];
                        acc[k] += v.w * row[i + 3];
                    }
                }
            }
        }
#pragma unroll 8
        for (; i < a.h1; ++i) {
            const T r = row[i];
#pragma unroll
            for (int k = 0; k < NB; ++k) acc[k] += __ldg(w[k] + i) * r;
        }
#pragma unroll
        for (int k = 0; k < NB; ++k)
            if (n + k < a.h2) sum += w3[n + k] * gelu_slow(acc[k], tab, a.two);
    }
    return sum;
}

// Shared memory of a team for 64 coalitions, in elements of the type:
// pre-activations [64][h1 + 1], those without the six low bits, what each of
// these adds, sums, values, and the list of rows.
constexpr int SLOW_FEW = 8;  // rows up to which a unit's products are split over lanes
__host__ __device__ constexpr int slow_elems(int h1) { return 64 * (h1 + 1) + 7 * h1 + SLOW_FEW * MAXH + 64 + 16; }
static_assert(2 * slow_elems(MAXH) * 8 <= Smem<true>::TAB && 4 * slow_elems(MAXH) * 4 <= Smem<false>::TAB,
              "two or four teams fit");
template <typename T>
__device__ __forceinline__ T *slow_values(T *scratch, int h1) { return scratch + 64 * (h1 + 1) + 7 * h1 + SLOW_FEW * MAXH; }

// The rows given (bit c: coalition S0 | c) of the 64 coalitions from S0 on and one
// background row in the arithmetic of the type, as masked_game_kernel has it, by
// a team of threads with a named barrier of its own: slow_values(scratch)[k] = f
// of the k-th of the rows.
template <typename T>
__device__ __forceinline__ void slow_group(const Args &a, const double *x, const double *base, int S0,
                                           unsigned long long rows, T *scratch, int tid, int team, int barrier,
                                           const ulonglong2 *tab) {
    const int warp = tid >> 5, lane = tid & 31, ld = a.h1 + 1, q = tid & 3;
    T *const pre = scratch, *const high = pre + 64 * ld, *const delta = high + a.h1, *const part = delta + 6 * a.h1;
    T *const value = slow_values(scratch, a.h1);
    unsigned char *const list = reinterpret_cast<unsigned char *>(value + 64);
    auto team_sync = [&] {
        __syncwarp();
        asm volatile("barrier.sync %0, %1;" ::"r"(barrier), "r"(team) : "memory");
    };
    const int n_rows = __popcll(rows);
    if (tid < 64 && ((rows >> tid) & 1)) list[__popcll(rows & ((1ull << tid) - 1))] = (unsigned char)tid;
    for (int j0 = 0; j0 < a.h1; j0 += team / 4) {
        const int j = j0 + (tid >> 2);
        double acc = 0.0;
        if (j < a.h1) {
            const double *w1 = a.W1 + j * a.d;
#pragma unroll 4
            for (int i = q; i < a.d; i += 4) acc += w1[i] * (i >= 6 && ((S0 >> i) & 1) ? x[i] : base[i]);
            for (int k = q; k < 6; k += 4) delta[k * a.h1 + j] = (T)(w1[k] * (x[k] - base[k]));
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if (q == 0 && j < a.h1) high[j] = (T)(a.b1[j] + acc);
    }
    team_sync();
    const int rows_on = team / a.h1, units_on = team - rows_on * a.h1;
    for (int c = tid / a.h1, j = tid - c * a.h1; c < n_rows;) {
        const int bits = list[c];
        T z = high[j];
#pragma unroll
        for (int k = 0; k < 6; ++k)
            if ((bits >> k) & 1) z += delta[k * a.h1 + j];
        pre[c * ld + j] = gelu_slow(z, tab, a.two);
        c += rows_on;
        j += units_on;
        if (j >= a.h1) {
            j -= a.h1;
            ++c;
        }
    }
    team_sync();
    int groups;
    if (n_rows <= SLOW_FEW) {
        // eight lanes share the products of a unit of layer 2
        groups = a.h2;
        const T *w2 = Weights<T>::w2(a), *b2 = Weights<T>::b2(a), *w3 = Weights<T>::w3(a);
        const int items = n_rows * a.h2;
        for (int i0 = 0; i0 < items; i0 += team / 8) {
            const int item = i0 + (tid >> 3), n = item / n_rows, c = item - n * n_rows;
            T acc = 0;
            if (item < items) {
#pragma unroll 4
                for (int i = tid & 7; i < a.h1; i += 8) acc += __ldg(w2 + n * a.h1 + i) * pre[c * ld + i];
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (item < items && (tid & 7) == 0) part[item] = acc;
        }
        team_sync();
        for (int item = tid; item < items; item += team) {
            const int n = item / n_rows;
            part[item] = w3[n] * gelu_slow(b2[n] + part[item], tab, a.two);
        }
    } else {
        // thread (coalition c, group g of units)
        groups = team / n_rows;
        const int c = tid % n_rows, g = tid / n_rows;
        if (g < groups)
            part[tid] = a.h2 >= 8 * groups ? slow_units<T, 4>(a, pre + c * ld, 4 * g, 4 * groups, tab)
                                           : slow_units<T, 1>(a, pre + c * ld, g, groups, tab);
    }
    team_sync();
    for (int k = warp; k < n_rows; k += team / 32) {
        T sum = 0;
        for (int g = lane; g < groups; g += 32) sum += part[g * n_rows + k];
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) value[k] = sum + (T)a.b3;
    }
    team_sync();
}

// Listed rows of one tile and background row (bit r of the mask: row r): thread
// r < 128 returns f of row r.  Each half of the CTA takes 64 rows.
template <typename T>
__device__ __noinline__ T slow_rows(const Args &a, int tile, int bgi, uint4 mask, unsigned char *smem) {
    T *const scratch = reinterpret_cast<T *>(smem);
    const ulonglong2 *tab = reinterpret_cast<const ulonglong2 *>(smem + Smem<true>::TAB);  // (float64)
    const int tile_shift = a.d - LOW, inst = tile >> tile_shift, S = (tile - (inst << tile_shift)) << LOW;
    const unsigned long long low = ((unsigned long long)mask.y << 32) | mask.x, high = ((unsigned long long)mask.w << 32) | mask.z;
    const int half = threadIdx.x / (THREADS / 2);
    if (half ? high : low)
        slow_group<T>(a, a.x + (long long)inst * a.d, a.bg + (long long)bgi * a.d, S | (half << 6), half ? high : low,
                      scratch + half * slow_elems(a.h1), threadIdx.x % (THREADS / 2), THREADS / 2, 1 + half, tab);
    __syncthreads();
    T result = 0;
    if (threadIdx.x < ROWS) {
        const int r = threadIdx.x & 63, h = threadIdx.x >> 6;
        const unsigned long long m = h ? high : low;
        if ((m >> r) & 1) result = slow_values(scratch + h * slow_elems(a.h1), a.h1)[__popcll(m & ((1ull << r) - 1))];
    }
    __syncthreads();
    return result;
}

// All values of tiles [t0, t1) of one instance (halves: of 64 coalitions of the
// one tile t0): teams of 128, 256 or 512 threads take 64 coalitions at a time, as
// the CTAs of masked_game_kernel do, each at its own pace.
template <typename T>
__device__ __noinline__ void slow_tiles(const Args &a, int t0, int t1, unsigned char *smem) {
    constexpr int BYTES = Smem<sizeof(T) == 8>::TAB;  // the activations' and W2's regions
    const int first = a.halves ? 2 * t0 + ((int)blockIdx.x & 1) : 2 * t0, end = a.halves ? first + 1 : 2 * t1;
    int teams = end - first >= 4 ? 4 : end - first;  // (1, 2 or 4: a tile has two halves)
    if (teams * slow_elems(a.h1) * (int)sizeof(T) > BYTES) teams = 2;
    const int team = THREADS / teams, k = threadIdx.x / team, tid = threadIdx.x - k * team;
    T *const scratch = reinterpret_cast<T *>(smem) + k * slow_elems(a.h1);
    const ulonglong2 *tab = reinterpret_cast<const ulonglong2 *>(smem + Smem<true>::TAB);  // (float64)
    const int tile_shift = a.d - LOW, inst = t0 >> tile_shift;
    const double *x = a.x + (long long)inst * a.d;
    for (int h = first + k; h < end; h += teams) {
        T sum = 0;
        for (int b = 0; b < a.n_bg; ++b) {
            slow_group<T>(a, x, a.bg + (long long)b * a.d, (h - (inst << (tile_shift + 1))) << 6, ~0ull, scratch, tid, team,
                          1 + k, tab);
            if (tid < 64) {
                const T f = slow_values(scratch, a.h1)[tid];
                sum = a.n_bg == 1 ? f : b == 0 ? (T)a.scale * f : sum + (T)a.scale * f;
            }
        }
        if (tid < 64) reinterpret_cast<T *>(a.v)[(long long)h * 64 + tid] = sum;
    }
    __syncthreads();
}

// The scales in place, besides the arrays in Smem.
struct Scales {
    int ok;        // the instance's rows may take the fixed point
    int version;   // of the arrays
    int row_span;  // rows down to 2^-row_span of the largest do
    int xmax, Q;   // float64: the most extra bits of a row in layer 2; fraction bits of layer 3 less a unit's
    int model_now, model_ok;         // the model's own scales are in place; they are of use
    float model_room;                // rounding of the type over what the digits add, at the model's bounds
    float model_al;                  // sum of those bounds in units of 2^E
    int const_x, const_Q;            // xmax and Q of the per-unit constants in place
    signed char model_e[MAXH];       // the model's exponents (127: a unit without weights)
    float redf[WARPS][10];
};

// Bounds of unit tid >> 2 over an instance's coalitions (x = null: for features
// of size C::TYPICAL): |z| <= beta, z <= zmax; lone: one feature leaves less to
// the others than the format spares.  Also the unit's |W1| (feature q + 4 k) and |b1|.
template <bool F64>
__device__ __forceinline__ void unit_bounds(const Args &a, const double *x, const float *most, float &beta, float &zmax,
                                            bool &lone, float (&w1)[8], float &b) {
    using C = Cfg<F64>;
    const int j = threadIdx.x >> 2, q = threadIdx.x & 3;
    const bool in = j < a.h1;
    float m[8];
    const double bias = in ? a.b1[j] : 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {  // (d <= 30; all loads in flight)
        const int i = q + 4 * k;
        const bool on = in && i < a.d;
        w1[k] = on ? magnitude(a.W1[(long long)j * a.d + i]) : 0.f;
        m[k] = !on ? 0.f : x ? fmaxf(magnitude(x[i]), most[i]) : C::TYPICAL;
    }
    float sum = 0.f, top = 0.f, rest = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float c = w1[k] * m[k];
        sum += c;  // (infinite or NaN if anything is)
        rest += fminf(c, top);
        top = fmaxf(top, c);
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        const float t2 = __shfl_xor_sync(0xffffffffu, top, o);
        rest += __shfl_xor_sync(0xffffffffu, rest, o) + fminf(top, t2);
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
        top = fmaxf(top, t2);
    }
    b = magnitude(bias);
    beta = sum + b;
    zmax = bias < 0.0 ? sum - b : sum + b;
    rest += b;
    lone = rest > 0.f && rest < C::LONE * top;
}

// Scales for an instance, or the model's own (x = null): exponents of the
// units of layer 1 and of the rows of W2 (scaled by its columns' exponents),
// formats of layers 2 and 3, and whether what the digits add stays below the
// type's own rounding (see the head of the file).  The whole CTA calls it.
template <bool F64>
__device__ __noinline__ void set_scales(const Args &a, const double *x, unsigned char *sm, Scales &sc) {
    using C = Cfg<F64>;
    using S = Smem<F64>;
    int *sE = reinterpret_cast<int *>(sm + S::SE), *sEw = reinterpret_cast<int *>(sm + S::EW);
    int *sFn = reinterpret_cast<int *>(sm + S::FN), *sMW = reinterpret_cast<int *>(sm + S::MW);
    float *sAl = reinterpret_cast<float *>(sm + S::PART);
    const int tid = threadIdx.x, lane = tid & 31, n = tid >> 2, q = tid & 3;
    float beta, zmax, w1[8], b1;
    bool lone;
    if (x) {
        // the model's scales serve where they hold the bounds with room to
        // spare, so that one set of W2's slices serves many instances
        unit_bounds<F64>(a, x, reinterpret_cast<const float *>(sm + S::MB), beta, zmax, lone, w1, b1);
        const bool bad = !(beta < 1e20f), dead = !(beta > 0.f) || zmax < -9.f;
        const float b = sc.model_e[n] == 127 ? 0.f : beta * pow2(-sc.model_e[n]);
        // (a unit's bound is in four threads); 1: not in the model's scales, 2: refused
        float v[2] = {bad || dead ? 0.f : 0.25f * b, bad || (lone && !dead) ? 2.f : 1.01f * b >= 1.f ? 1.f : 0.f};
        block_reduce<2, 1>(v, sc.redf);
        const bool refused = v[1] == 2.f;
        const bool fits = v[1] == 0.f && sc.model_ok && v[0] * sc.model_room >= sc.model_al;
        if (refused || (fits && sc.model_now)) {
            if (tid == 0) sc.ok = !refused;
            __syncthreads();
            return;
        }
        if (fits) x = nullptr;  // back to the model's
    }
    const bool model = !x;
    if (model) {
        unit_bounds<F64>(a, nullptr, nullptr, beta, zmax, lone, w1, b1);
        if (zmax < -9.f) zmax = 0.f;  // dead for some instances only
    }
    if (tid < 32) sMW[tid] = 0;

    bool bad = !(beta < 1e20f);
    const bool dead = !(beta > 0.f) || zmax < -9.f;  // no activation that counts
    const int e = max(dead || bad ? C::EMIN : exp_above(1.01f * beta), C::EMIN);
    bad |= e > C::EMAX;
    const float al = dead || bad ? 0.f : beta * pow2(-e);
    if (q == 0) {
        sE[n] = (min(e, C::EMAX) + 64) | (dead ? kDead : 0);
        sAl[n] = al;
        if (sc.version == 0) sc.model_e[n] = dead ? 127 : (signed char)min(e, C::EMAX);
    }
    __syncthreads();
    // the most that a feature of size 1 (at d: that b1) gives an activation, in units of 2^E
    const float unit = dead || bad ? 0.f : pow2(-e);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        float m = w1[k] * unit;
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane < 4 && q + 4 * k < a.d) atomicMax(sMW + q + 4 * k, __float_as_int(m));  // none is negative
    }
    // (a negative bias lifts no activation; GELU is never below -0.17)
    const int b_most = __reduce_max_sync(0xffffffffu, __float_as_int((zmax < beta ? fminf(b1, 0.18f) : b1) * unit));
    if (lane == 0) atomicMax(sMW + a.d, b_most);

    float wmax = 0.f, wsum = 0.f, nat = 0.f, top = 0.f;
    int count = 0;
    double bias2 = 0.0, weight3 = 0.0;
    if (n < a.h2) {
        bias2 = a.b2[n];
        weight3 = a.W3[n];
#pragma unroll 8
        for (int j = q; j < a.h1; j += 4) {
            const float m = magnitude(a.W2[(long long)n * a.h1 + j]);
            bad |= !(m < 1e20f);
            const float w = (sE[j] & kDead) ? 0.f : m * pow2((sE[j] & 255) - 64), c = w * sAl[j];
            wmax = fmaxf(wmax, w);
            wsum += w;
            nat += c;
            top = fmaxf(top, c);
            count += c > 0.f;
        }
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        wmax = fmaxf(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
        top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
        wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
        nat += __shfl_xor_sync(0xffffffffu, nat, o);
        count += __shfl_xor_sync(0xffffffffu, count, o);
    }
    const float b2 = magnitude(bias2), w3 = magnitude(weight3);
    bad |= !(b2 < 1e20f) || !(w3 < 1e18f) || (weight3 != 0.0 && w3 < 1e-18f) || !(wsum < 1e18f);
    const float zb = 1.02f * wsum + b2;
    const bool live = w3 > 0.f && !((bias2 < 0.0 ? 1.02f * wsum - b2 : zb) < -9.f);
    const int ze = exp_above(zb);
    int ew = max(exp_above(1.01f * wmax), -60), fn = 0, xmax = 0, x_b2 = 0;
    if constexpr (F64) {
        // a row whose activations are 2^-x of the largest keeps x more bits of
        // layer 2 where b2 allows it and the format, of 62 bits, has them
        float less[2] = {live && b2 > 0.f ? (float)max(0, C::SPAN - max(0, ze - exp_above(b2))) : 0.f,
                         live ? (float)max(0, C::SPAN - max(0, 1 + ze)) : 0.f};
        block_reduce<2, 0>(less, sc.redf);
        x_b2 = C::SPAN - (int)less[0];
        xmax = min(x_b2, C::SPAN - (int)less[1]);
        fn = live ? min(61 - ze, 62 - xmax) : 62 - xmax;
        ew = max(ew, 45 - fn);
        bad |= live && ze > 18;
    } else {
        bad |= ew > 60;
    }
    if (q == 0) {
        sEw[n] = live ? ew : kDead;
        if constexpr (F64) sFn[n] = fn;
    }
    // the digits of W2 end 2^-57 (float64) or 2^-33 (float32) below the largest of
    // a row; the type itself loses 2^-54 or 2^-25 of each product and more in sums
    const bool on = q == 0 && live, several = on && count > 1;
    const float k_row = C::EVEN * fmaxf(12.f, 3.f * sqrtf((float)count));
    constexpr int NV = F64 ? 10 : 3, NS = F64 ? 8 : 3;
    float v[NV];
    v[0] = several ? w3 * wmax * (float)(count - 1) : 0.f;
    v[1] = several ? w3 * k_row * (nat - top) : 0.f;
    v[2] = q == 0 ? al : 0.f;
    if constexpr (F64) {
        v[3] = on ? w3 * zb : 0.f;                        // what a unit can give layer 3
        v[4] = on ? w3 * fminf(1.f, 0.125f * zb) : 0.f;   // and about gives
        v[5] = on ? w3 * w3 : 0.f;
        v[6] = on ? 1.f : 0.f;
        v[7] = q == 0 && !dead ? (float)(e + 4096) : 0.f;  // exponents and (4096 each) number of live units
        v[8] = on ? w3 * pow2(61 - fn) : 0.f;
        v[9] = on ? w3 * zb : 0.f;
    }
    block_reduce<NV, NS>(v, sc.redf);
    bool ok = !__syncthreads_or(bad);
    if (tid == 0) {
        const float room = v[0] > 0.f ? v[1] / v[0] : 1e30f;
        sc.row_span = C::SPAN;
        sc.xmax = sc.Q = 0;
        if constexpr (F64) {
            const float units = v[6], live_units = floorf(v[7] * (1.f / 4096.f));
            if (units > 1.f)  // W3's 53 bits of its largest against the units' own
                ok = ok && v[8] * (units - 1.f) <= 2.f * fmaxf(12.f, 3.f * sqrtf(units)) * (v[3] - v[9]);
            // the table's 2^-59 against what double loses of what the units give
            const float mu = v[5] > 0.f ? 128.f * v[4] * rsqrtf(v[5] * units) : 1e30f;
            const int e_mean = live_units > 0.f ? (int)floorf((v[7] - 4096.f * live_units) / live_units) : C::SPAN;
            sc.row_span = min(min(C::SPAN, e_mean + 3), exp_above(mu) - 2);
            if (xmax < x_b2) sc.row_span = min(sc.row_span, xmax + 1);
            ok = ok && mu >= 8.f;
            sc.xmax = xmax;
            sc.Q = 114 - max(exp_above(v[8]), -60);
        }
        if (sc.version == 0) {
            sc.model_ok = ok;
            sc.model_room = room;
            sc.model_al = v[2];
        }
        sc.version += 1;
        sc.model_now = model;
        sc.ok = ok && (model || room >= 1.f);
    }
    __syncthreads();
}

template <bool F64>
__global__ void __launch_bounds__(THREADS, 1) masked_game_split_kernel(const __grid_constant__ Args a) {
    using C = Cfg<F64>;
    using S = Smem<F64>;
    using T = typename std::conditional<F64, double, float>::type;
    constexpr int NS = C::NS, ND = C::ND, NW = C::NW, BITS = C::BITS, CPT = C::CPT, CHUNKS = S::CHUNKS;
    extern __shared__ __align__(1024) unsigned char sm_raw[];
    const uint32_t raw = smem_u32(sm_raw);
    unsigned char *sm = sm_raw + (((raw + 1023) & ~1023u) - raw);
    unsigned char *smA = sm + S::A, *smW = sm + S::W;
    ulonglong2 *tab = reinterpret_cast<ulonglong2 *>(sm + S::TAB);
    // layer-1 pre-activations: sums of integers with 62 fraction bits of the
    // unit's 2^E; float32 takes them up from bits 3 .. 6 on as floats
    using P = typename std::conditional<F64, i64, float>::type;
    P *PH = reinterpret_cast<P *>(sm + S::PH);
    i64 *DL = reinterpret_cast<i64 *>(sm + S::DL);
    float *DF = reinterpret_cast<float *>(sm + S::DF);
    int *sE = reinterpret_cast<int *>(sm + S::SE), *sEw = reinterpret_cast<int *>(sm + S::EW);
    int *sFn = reinterpret_cast<int *>(sm + S::FN);
    using R = typename std::conditional<F64, signed char, float>::type;
    R *sEr = reinterpret_cast<R *>(sm + S::ER);
    int *sCs = reinterpret_cast<int *>(sm + S::CS), *sCe = reinterpret_cast<int *>(sm + S::CE);
    const float *sMW = reinterpret_cast<const float *>(sm + S::MW);
    int *sMB = reinterpret_cast<int *>(sm + S::MB);
    __shared__ __align__(8) uint64_t mbar, ph_ready, part_ready;  // MMAs done; tables made; row sums written
    __shared__ uint32_t tmem_sh;
    __shared__ Scales sc;
    __shared__ __align__(16) unsigned sFlag[2][4];  // rows left to slow_rows, double-buffered

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        mbar_init(smem_u32(&mbar), 1);
        mbar_init(smem_u32(&ph_ready), WARPS);
        mbar_init(smem_u32(&part_ready), WARPS * 3 / 4);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_sh)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
        sMB[lane] = 0;
        if (lane == 0) sc.version = 0;
    }
    if constexpr (F64)
        for (int i = tid; i < TAB_ROWS * 2; i += THREADS) tab[i] = (&g_gelu_table[0][0])[i];
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_sh;
    if (lane < a.d) {
        float m = 0.f;
        for (int k = warp; k < a.n_bg; k += WARPS) m = fmaxf(m, magnitude(a.bg[(long long)k * a.d + lane]));
        atomicMax(sMB + lane, __float_as_int(m));  // none is negative
    }
    __syncthreads();
    const uint32_t a_base = smem_u32(smA), w_base = smem_u32(smW);  // below 2^18: descriptors add up

    const int n_kc = (a.h1 + KC - 1) / KC, n_nh = (a.h2 + NW - 1) / NW;
    const int tile_shift = a.d - LOW;
    // (2^31 tiles would be 2^38 values)
    const int t_begin = a.halves ? (int)blockIdx.x >> 1 : (int)(a.n_tiles * blockIdx.x / gridDim.x);
    const int t_end = a.halves ? t_begin + 1 : (int)(a.n_tiles * (blockIdx.x + 1) / gridDim.x);
    // the rows this CTA gives out, by quarters
    auto own = [&](int quarter) { return !a.halves || (quarter >> 1) == (blockIdx.x & 1) ? ~0u : 0u; };
    const bool own_row = tid < ROWS && own(warp);
    uint32_t parity = 0, ph_parity = 0, part_parity = 0;
    bool failed = false;  // a bounded wait ran out (of this warp until the CTA's barrier)
    // a warp's arrival and wait (lane 0 for the warp, bounded)
    auto arrive = [&](uint64_t *bar) {
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
        __syncwarp();
    };
    auto wait = [&](uint64_t *bar, uint32_t &phase) {
        // every lane polls, so that the warp stays together
        failed |= !__all_sync(0xffffffffu, mbar_wait(smem_u32(bar), phase));
        __syncwarp();
        phase ^= 1u;
    };

    set_scales<F64>(a, nullptr, sm, sc);

    // epilogue state: the accumulators of the pass in flight, its row sums so
    // far, and (threads < 128) the sum over background rows of row tid
    i64 zi[F64 ? CPT : 1];
    float zf[F64 ? 1 : CPT];
    i64 acc_hh = 0, acc_hl = 0, acc_lh = 0, acc_ll = 0;
    float acc_f = 0.f, acc_f1 = 0.f;  // even and odd columns
    T vsum = 0;
    bool slow = false;  // row tid of the tile and background row came from slow_rows
    enum : int { kWaiting = 1, kLastPass = 2, kFirstBg = 4, kLastBg = 8, kSlow = 16 };
    int pend = 0;       // the pass in flight
    int pend_x = 0, pend_tile = 0;

    // epilogue: thread (row, quarter of the pass's columns), in whole loads of 8
    const int n_col = min(NW, a.h2);
    const int cpt = min(CPT, ((n_col + 31) >> 5) << 3);
    const int erow = 32 * (warp & 3) + lane, ecol = (warp >> 2) * cpt;

    auto emit = [&](T f, bool first, bool last, int tile) {  // threads < 128
        if (a.n_bg == 1)
            vsum = f;
        else
            vsum = first ? (T)a.scale * f : vsum + (T)a.scale * f;
        if (last && own_row) reinterpret_cast<T *>(a.v)[(long long)tile * ROWS + tid] = vsum;
    };
    auto emit_pending = [&](T f) {  // a slow row's value is in already
        if (!(pend & kSlow)) emit(f, pend & kFirstBg, pend & kLastBg, pend_tile);
    };

    // Layers 2 (GELU) and 3 of the drained accumulators.
    auto finish_pending = [&]() {
        if (!(pend & kWaiting)) return;
        pend &= ~kWaiting;
        if constexpr (F64) {
            const i64 *b2q = reinterpret_cast<const i64 *>(sm + S::COL) + ecol;
            const int2 *w3q = reinterpret_cast<const int2 *>(sm + S::COL + NW * 8) + ecol;
            const int *cs = sCs + ecol, down = sc.const_x - pend_x;
            // eight columns an iteration from the front of the register array,
            // which then moves up (a run-time loop keeps the code short)
#pragma unroll 1
            for (int c = 0; c < cpt; c += 8) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const i64 g = gelu_fixed(zi[k] + shr(b2q[c + k], down), cs[c + k] - pend_x, tab, a.two);
                    // g times W3 = wh 2^27 + wl, exact: the parts' products are at most
                    // 2^57 and there are at most 32 of each
                    const int2 w = w3q[c + k];
                    const int gh = hi32(g), gl = (int)(lo32(g) >> 1);
                    acc_hh = mad_wide(gh, w.x, acc_hh);
                    acc_hl = mad_wide(gh, w.y, acc_hl);
                    acc_lh = mad_wide(gl, w.x, acc_lh);
                    acc_ll = mad_wide(gl, w.y, acc_ll);
                }
#pragma unroll
                for (int k = 0; k + 8 < CPT; ++k) zi[k] = zi[k + 8];
            }
        } else {
            const float4 *p2 = reinterpret_cast<const float4 *>(sm + S::COL) + ecol;
#pragma unroll 1
            for (int c = 0; c < cpt; c += 8) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float4 p = p2[c + k];  // b2, W3, scale of W2's row
                    float &acc = k & 1 ? acc_f1 : acc_f;
                    acc = fmaf(p.y, gelu_fast(fmaf(zf[k], p.z, p.x)), acc);
                }
#pragma unroll
                for (int k = 0; k + 8 < CPT; ++k) zf[k] = zf[k + 8];
            }
        }
        if (pend & kLastPass) {
            // sum over the four column groups of a row (group 0 is threads < 128)
            const int group = warp >> 2;
            if constexpr (F64) {
                longlong2 *pt = reinterpret_cast<longlong2 *>(sm + S::PART);
                __int128 w = ((__int128)acc_hh << 59) + ((__int128)acc_hl << 32) + ((__int128)acc_lh << 28) +
                             ((__int128)acc_ll << 1);
                if (group) {
                    pt[(group - 1) * ROWS + erow] = make_longlong2((i64)(u64)w, (i64)(w >> 64));
                    arrive(&part_ready);
                } else {
                    wait(&part_ready, part_parity);
                    for (int k = 0; k < 3; ++k) {
                        const longlong2 o = pt[k * ROWS + tid];
                        w += (__int128)(((unsigned __int128)(u64)o.y << 64) | (u64)o.x);
                    }
                    // a double: its 64 leading bits (the rest is below its rounding), scaled back
                    const bool neg = w < 0;
                    const unsigned __int128 u = neg ? (unsigned __int128)0 - (unsigned __int128)w : (unsigned __int128)w;
                    const u64 hi = (u64)(u >> 64), lo = (u64)u;
                    const int lz = hi ? __clzll((i64)hi) : 64;
                    const u64 top = lz == 0 ? hi : lz == 64 ? lo : (hi << lz) | (lo >> (64 - lz));
                    const double s = (double)(neg ? -(i64)(top >> 1) : (i64)(top >> 1));
                    // units 2^-(Q + x), and 2^(65 - lz) of them (2 when all is in the low word)
                    const int e = 65 - lz - (sc.const_Q + pend_x);
                    emit_pending(s * __longlong_as_double((i64)(1023 + e) << 52) + a.b3);
                }
            } else {
                float *pf = reinterpret_cast<float *>(sm + S::PART);
                acc_f += acc_f1;
                if (group) {
                    pf[(group - 1) * ROWS + erow] = acc_f;
                    arrive(&part_ready);
                } else {
                    wait(&part_ready, part_parity);
                    const float s = (acc_f + pf[tid]) + (pf[ROWS + tid] + pf[2 * ROWS + tid]);
                    emit_pending(s + (float)a.b3);
                }
            }
            acc_hh = acc_hl = acc_lh = acc_ll = 0;
            acc_f = acc_f1 = 0.f;
        }
    };

    // ---- the walk over (tile, background row, pass over layer 2, K chunk) ----
    int t = t_begin;
    int bgi = 0, nh = 0, kc = 0;
    int inst_now = -1, bg_now = -1;  // the instance and background row of the scales and tables in place
    int const_nh = -1, const_version = -1;  // what the epilogue's per-unit constants were made for
    // the chunk of them that DL, dhigh and base0 hold (float32: a bit for each that is held)
    constexpr int NO_CHUNK = F64 ? -1 : 0;
    int chunk_key = NO_CHUNK;
    int w_key = -1, w_version = -1;  // (nh, kc) of the resident slices of W2 (float32: the chunks made)
    int rbuf = 0;              // buffer of sEr and sFlag of the tile and background row
    bool ok = false;
    i64 dhigh[CHUNKS][3] = {}, base0[CHUNKS] = {};
    // layer-1 tables: lanes 8 v + part of a warp have unit 4 warp + v of the chunk
    const int part = lane & 7, jj = 4 * warp + (lane >> 3);
    // Ahead of a call: a finished pass and the tables leave nothing in registers
    // over it (the tables are made again) but the sums of a tile's passes so far.
    auto forget = [&]() {
#pragma unroll
        for (int k = 0; k < (F64 ? CPT : 1); ++k) zi[k] = 0;
#pragma unroll
        for (int k = 0; k < (F64 ? 1 : CPT); ++k) zf[k] = 0.f;
#pragma unroll
        for (int c = 0; c < CHUNKS; ++c) {
            base0[c] = 0;
#pragma unroll
            for (int k = 0; k < 3; ++k) dhigh[c][k] = 0;
        }
        chunk_key = NO_CHUNK;
    };

    // The layer-1 tables of the step at (t, bgi, kc), after every warp is done
    // with those before: scales when the instance changes, row scales with the
    // tile or background row, then PH[e][j] = the empty coalition's
    // pre-activation + the high features' + those of bits 3 .. 6 (pattern e).
    auto prepare_step = [&]() {
        const int inst = t >> tile_shift, S_high = (t - (inst << tile_shift)) << LOW;
        const double *x = a.x + (long long)inst * a.d;
        const double *base = a.bg + (long long)bgi * a.d;
        const bool new_row = inst_now != inst || bg_now != bgi;
        if (inst_now != inst) {
            finish_pending();
            forget();
            inst_now = inst;
            set_scales<F64>(a, x, sm, sc);
            ok = sc.ok;
        }
        if (bg_now != bgi) chunk_key = NO_CHUNK;
        bg_now = bgi;
        const bool first = nh == 0 && kc == 0;
        if (first) rbuf ^= 1;
        if (!ok) return;
        if (first && warp >= WARPS - 4) {
            // a row's scale: what its features and b1 can give any unit, in units of
            // 2^E; the low features' part once per background row (each of the four
            // warps writes the same float2s and reads its own)
            const int quarter = warp - (WARPS - 4), r = 32 * quarter + lane;
            float2 *mx = reinterpret_cast<float2 *>(sm + S::MX);
            float *low = reinterpret_cast<float *>(sm + S::RL) + r;
            if (new_row) {
                const float m = lane < a.d ? sMW[lane] : 0.f;
                mx[lane] = lane < a.d ? make_float2(m * magnitude(x[lane]), m * magnitude(base[lane])) : make_float2(0.f, 0.f);
                __syncwarp();
                float sum = sMW[a.d];
#pragma unroll
                for (int k = 0; k < LOW; ++k) sum += ((r >> k) & 1) ? mx[k].x : mx[k].y;
                *low = sum;
            }
            const float2 f = mx[lane];
            float sum = lane >= LOW ? (((S_high >> lane) & 1) ? f.x : f.y) : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            sum += *low;
            // (a row of zeros has any scale)
            const int e = sum > 0.f ? min(0, exp_above(1.01f * sum)) : 0;
            const unsigned flags = __ballot_sync(0xffffffffu, -e > sc.row_span) & own(quarter);
            const int e_row = max(e, -sc.row_span);
            if constexpr (F64)
                sEr[rbuf * ROWS + r] = (R)e_row;
            else
                sEr[rbuf * ROWS + r] = pow2(31 - e_row);
            if (lane == 0) sFlag[rbuf][quarter] = flags;
        }
        const int j = kc * KC + jj;
        const bool in = j < a.h1 && !(sE[j] & kDead);
        const int slot = F64 ? 0 : kc;
        const int ej = (sE[j] & 255) - 64;
        const float down = F64 ? 0.f : pow2(ej - 62);
        i64 *dl = DL + slot * (LOW * KC) + jj;
        if (F64 ? chunk_key != kc : ((chunk_key >> kc) & 1) == 0) {
            // every feature's contribution when it joins the coalition: the low
            // seven in shared memory, the high ones (at most three per lane) in
            // registers; and the empty coalition's sum
            chunk_key = F64 ? kc : chunk_key | (1 << kc);
            const int f1 = 62 - ej;
            const double *w1 = a.W1 + (long long)(in ? j : 0) * a.d;
            i64 z0 = 0, dlow = 0, dh[3];
            if (in && part == 7) z0 = fix(a.b1[j], f1);
            if (in && part < LOW) {
                z0 = fix(w1[part] * base[part], f1);
                dlow = fix(w1[part] * x[part], f1) - z0;
            }
            if (part < LOW) {
                dl[part * KC] = dlow;
                if (!F64 && part < 3) DF[(slot * 3 + part) * KC + jj] = (float)dlow * down;
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int i = LOW + part + 8 * k;
                dh[k] = 0;
                if (in && i < a.d) {
                    const i64 z = fix(w1[i] * base[i], f1);
                    z0 += z;
                    dh[k] = fix(w1[i] * x[i], f1) - z;
                }
            }
#pragma unroll
            for (int c = 0; c < CHUNKS; ++c)
                if (c == slot) {
                    base0[c] = z0;
#pragma unroll
                    for (int k = 0; k < 3; ++k) dhigh[c][k] = dh[k];
                }
            __syncwarp();
        }
        i64 s = slot ? base0[CHUNKS - 1] : base0[0];
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if ((S_high >> (LOW + part + 8 * k)) & 1) s += slot ? dhigh[CHUNKS - 1][k] : dhigh[0][k];
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        // entries part and part + 8
#pragma unroll
        for (int m = 0; m < 3; ++m)
            if ((part >> m) & 1) s += dl[(3 + m) * KC];
        if constexpr (F64) {
            PH[part * KC + jj] = s;
            PH[(part + 8) * KC + jj] = s + dl[6 * KC];
        } else {
            PH[part * KC + jj] = (float)s * down;
            PH[(part + 8) * KC + jj] = (float)(s + dl[6 * KC]) * down;
        }
    };
    auto next_step = [&]() {  // the background row or tile after this one
        nh = kc = 0;
        if (++bgi == a.n_bg) {
            bgi = 0;
            ++t;
        }
    };

    // One barrier of the whole CTA per step (before its MMAs are issued); a warp
    // otherwise goes on from the pass before to the next layer 1 by itself.
    if (t < t_end) {
        prepare_step();
        arrive(&ph_ready);
    }
    while (t < t_end) {
        wait(&ph_ready, ph_parity);
        if (nh == 0 && kc == 0) {
            slow = false;
            if (!ok) {
                // (after a barrier: see the end of the walk)
                if (__syncthreads_or(failed ? 1 : 0)) {
                    failed = true;
                    break;
                }
                finish_pending();
                forget();
                const int stop = min(t_end, ((t >> tile_shift) + 1) << tile_shift);
                slow_tiles<T>(a, t, stop, smA);
                w_version = 0;  // W2's slices are overwritten
                t = stop;
                if (t < t_end) {
                    prepare_step();
                    arrive(&ph_ready);
                }
                continue;
            }
            const uint4 flags = *reinterpret_cast<const uint4 *>(sFlag[rbuf]);
            if (flags.x | flags.y | flags.z | flags.w) {
                if (__syncthreads_or(failed ? 1 : 0)) {
                    failed = true;
                    break;
                }
                finish_pending();
                forget();
                const T f = slow_rows<T>(a, t, bgi, flags, smA);
                const unsigned quarter = warp == 0 ? flags.x : warp == 1 ? flags.y : warp == 2 ? flags.z : flags.w;
                slow = warp < 4 && ((quarter >> lane) & 1u);
                if (slow) emit(f, bgi == 0, bgi == a.n_bg - 1, t);
                if (2 * slow_elems(a.h1) * (int)sizeof(T) > NS * SLICE_A) w_version = 0;
                if (flags.x == own(0) && flags.y == own(1) && flags.z == own(2) && flags.w == own(3)) {
                    next_step();
                    if (t < t_end) {
                        prepare_step();
                        arrive(&ph_ready);
                    }
                    continue;
                }
            }
        }
        const R *er = sEr + rbuf * ROWS;
        // ---- layer 1: units 2u, 2u + 1 of the chunk; a warp has rows 8 warp ..
        // 8 warp + 7, split over its lanes when the chunk has at most 32 or 16
        // units; a lane walks its rows in pairs (bit 0) ----
        {
            const int units = min(KC, a.h1 - kc * KC);
            const int lg = units <= 16 ? 3 : units <= 32 ? 4 : 5, nb = lg - 2;
            const int u = lane & ((1 << lg) - 1), sub = lane >> lg;
            const P *ph = PH + warp * KC + 2 * u;
            P pa = ph[0], pb = ph[1], da[3], db[3];
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                if constexpr (F64) {
                    da[m] = DL[m * KC + 2 * u];
                    db[m] = DL[m * KC + 2 * u + 1];
                } else {
                    da[m] = DF[(kc * 3 + m) * KC + 2 * u];
                    db[m] = DF[(kc * 3 + m) * KC + 2 * u + 1];
                }
                if (m >= nb && ((sub >> (m - nb)) & 1)) {
                    pa += da[m];
                    pb += db[m];
                }
            }
            const int row0 = 8 * warp + (sub << nb);
            const int2 e2 = *reinterpret_cast<const int2 *>(sE + kc * KC + 2 * u);
            const int ea = (e2.x & 255) - 64, eb = (e2.y & 255) - 64;
            const float ua = F64 ? 0.f : pow2(-ea), ub = F64 ? 0.f : pow2(-eb);
            auto put = [&](P za, P zb, int row) {
                unsigned char *dst = smA + pair_offset(row, u);
                if constexpr (F64) {
                    // rounded to 55 fraction bits of 2^(E + the row's exponent) and biased
                    const int sh = 7 + er[row];
                    const i64 c = join((lo32(BIAS7) << sh) | (1u << (sh - 1)),
                                       (int)__funnelshift_l(lo32(BIAS7), (unsigned)hi32(BIAS7), sh));
                    put_digits(dst, SLICE_A, (u64)shr(gelu_fixed(za, ea, tab, a.two) + c, sh),
                               (u64)shr(gelu_fixed(zb, eb, tab, a.two) + c, sh));
                } else {
                    const float up = er[row];
                    put_digits(dst, SLICE_A, (unsigned)__float2int_rn(gelu_fast(za) * ua * up) + BIAS4,
                               (unsigned)__float2int_rn(gelu_fast(zb) * ub * up) + BIAS4);
                }
            };
#pragma unroll 1
            for (int q = 0; q < (1 << (nb - 1)); ++q) {
                P ca = 0, cb = 0;  // (the small terms first: a float32 z has one rounding of its size)
                if (q & 1) {
                    ca = da[1];
                    cb = db[1];
                }
                if (q & 2) {
                    ca += da[2];
                    cb += db[2];
                }
                const int row = row0 + 2 * q;
                put(pa + ca, pb + cb, row);
                put(pa + (ca + da[0]), pb + (cb + db[0]), row + 1);
            }
        }
        // ---- the slices of W2 for (nh, kc) (float64: one chunk is held;
        // float32: both, made with the first tile of new scales) ----
        if (w_version != sc.version) {
            w_version = sc.version;
            w_key = -1;
        }
        if (F64 ? w_key != nh * n_kc + kc : w_key < kc) {
            w_key = F64 ? nh * n_kc + kc : kc;
            unsigned char *w_dst = smW + (F64 ? 0 : kc * (NS * NW * 128));
            const int u = lane, j0 = kc * KC + 2 * u;
            const int2 e2 = *reinterpret_cast<const int2 *>(sE + j0);
            const int ea = BITS - 64 + (e2.x & 255), eb = BITS - 64 + (e2.y & 255);
            const bool in_a = j0 < a.h1 && !(e2.x & kDead), in_b = j0 + 1 < a.h1 && !(e2.y & kDead);
            for (int n = warp; n < NW; n += WARPS) {
                const int gn = nh * NW + n, ew = sEw[gn];
                i64 wa = 0, wb = 0;
                if (gn < a.h2 && ew != kDead) {
                    const double *w = a.W2 + (long long)gn * a.h1;
                    if (in_a) wa = fix(w[j0], ea - ew);
                    if (in_b) wb = fix(w[j0 + 1], eb - ew);
                }
                if constexpr (F64)
                    put_digits(w_dst + pair_offset(n, u), NW * 128, (u64)wa + BIAS7, (u64)wb + BIAS7);
                else
                    put_digits(w_dst + pair_offset(n, u), NW * 128, (unsigned)wa + BIAS4, (unsigned)wb + BIAS4);
            }
        }
        // ---- layer 2's products on the tensor cores ----
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (__syncthreads_or(failed ? 1 : 0)) {
            failed = true;
            break;
        }
        if (warp == 0 && ttfsi_gemm::elect_one()) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int n_k16 = (min(KC, a.h1 - kc * KC) + 15) >> 4;
            const uint64_t da = smem_desc(a_base), dw = smem_desc(w_base + (F64 ? 0 : kc * (NS * NW * 128)));
            // digit i of the activations times up to 256 / NW neighbouring digits of
            // W2 in one MMA: their slices follow each other in shared memory as
            // their diagonals do in tensor memory.  Unrolled, so that each MMA costs
            // this thread a few instructions: the other warps end up waiting for it.
#pragma unroll
            for (int i = 0; i < NS; ++i) {
                const int j_end = NS < ND - i ? NS : ND - i;
#pragma unroll
                for (int j = 0; j < j_end; j += 256 / NW) {
                    const int n = 256 / NW < j_end - j ? 256 / NW : j_end - j;
                    // diagonal NS is written first by digits (1, NS - 1): on its own
                    const bool split = ND > NS && i == 1 && j + n == NS;
#pragma unroll
                    for (int part_no = 0; part_no < (split ? 2 : 1); ++part_no) {
                        const int j0 = part_no ? NS - 1 : j, m = part_no ? 1 : split ? n - 1 : n;
                        if (m == 0) continue;
                        const bool opens = i == 0 || (split && part_no == 1);
                        // FP32 accumulators, FP16 operands, both K-major, M = 128, N = m NW
                        const uint32_t idesc = (1u << 4) | ((uint32_t)(m * NW >> 3) << 17) | ((uint32_t)(ROWS >> 4) << 24);
#pragma unroll
                        for (int k16 = 0; k16 < 4; ++k16)
                            if (k16 < n_k16)
                                mma_f16(tmem + (i + j0) * NW, da + ((i * SLICE_A + k16 * 32) >> 4),
                                        dw + ((j0 * (NW * 128) + k16 * 32) >> 4), idesc,
                                        opens && k16 == 0 ? (kc > 0 ? 1u : 0u) : 1u);
                    }
                }
            }
            mma_commit(smem_u32(&mbar));
        }
        // ---- meanwhile the tables of the next step and the pass before ----
        const bool last_kc = kc == n_kc - 1;
        const int c_nh = nh, c_bg = bgi, c_rbuf = rbuf;
        const int c_t = t;
        if (last_kc && (const_nh != nh || const_version != sc.version)) {
            // per-unit constants of this pass's epilogue, while its scales are in place
            const_nh = nh;
            const_version = sc.version;
            finish_pending();
            __syncthreads();
            if (tid == 0) {
                sc.const_x = sc.xmax;
                sc.const_Q = sc.Q;
            }
            if (tid < NW) {
                const int gn = nh * NW + tid, ew = sEw[gn];
                const bool in = gn < a.h2 && ew != kDead;
                if constexpr (F64) {
                    const int fn = sFn[gn];
                    reinterpret_cast<i64 *>(sm + S::COL)[tid] = in ? fix(a.b2[gn], fn + sc.xmax) : 0;
                    const i64 w = in ? fix(a.W3[gn], sc.Q - fn) : 0;  // wh 2^27 + wl, |wl| <= 2^26
                    const int wh = (int)((w + (1ll << 26)) >> 27);
                    reinterpret_cast<int2 *>(sm + S::COL + NW * 8)[tid] = make_int2(wh, (int)(w - ((i64)wh << 27)));
                    sCs[tid] = 62 - fn;
                    sCe[tid] = in ? ew + fn - 38 : 7;
                } else {
                    reinterpret_cast<float4 *>(sm + S::COL)[tid] =
                        in ? make_float4((float)a.b2[gn], (float)a.W3[gn], pow2(ew), 0.f) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
            __syncthreads();
        }
        if (!last_kc) {
            ++kc;
        } else if (nh < n_nh - 1) {
            kc = 0;
            ++nh;
        } else {
            next_step();
        }
        if (t < t_end) {
            prepare_step();
            arrive(&ph_ready);
        }
        finish_pending();
        wait(&mbar, parity);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (!last_kc) continue;
        // ---- drain the accumulators of this pass into registers ----
        const int e_row = F64 ? (int)sEr[c_rbuf * ROWS + erow] : 0, x_row = min(-e_row, sc.const_x);
        // float32: 2^(e - 14), from the exponents of 2^(31 - e)
        const float zscale = F64 ? 0.f : __uint_as_float((271u << 23) - __float_as_uint((float)sEr[c_rbuf * ROWS + erow]));
        const uint32_t lane_base = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)ecol;
        if constexpr (F64) {
#pragma unroll
            for (int c = 0; c < CPT; c += 8) {
                if (c >= cpt) break;
                i64 up[8], low[8];
#pragma unroll
                for (int dg = 0; dg < 8; ++dg) {
                    uint32_t r[8];
                    tmem_ld8(lane_base + dg * NW + c, r);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int q = __float2int_rn(__uint_as_float(r[k]));
                        i64 &acc = dg < 4 ? up[k] : low[k];
                        acc = (dg & 3) ? mad_wide(q, a.unit[dg & 3], acc) : mul_wide(q, a.unit[0]);
                    }
                }
                // the parts are in units of 2^(e + ew - 38) and 2^(e + ew - 70), e the row's exponent;
                // the format of layer 2 is the unit's f and the row's x bits
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int sl = sCe[ecol + c + k] + e_row + x_row;
                    zi[c + k] = join(lo32(up[k]) << sl, (int)__funnelshift_l(lo32(up[k]), (unsigned)hi32(up[k]), sl)) +
                                shr(low[k], 32 - sl);
                }
            }
        } else {
#pragma unroll
            for (int c = 0; c < CPT; c += 8) {
                if (c >= cpt) break;
#pragma unroll
                for (int dg = 3; dg >= 0; --dg) {
                    uint32_t r[8];
                    tmem_ld8(lane_base + dg * NW + c, r);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        zf[c + k] = dg == 3 ? __uint_as_float(r[k]) : fmaf(zf[c + k], 0.00390625f, __uint_as_float(r[k]));
                }
#pragma unroll
                for (int k = 0; k < 8; ++k) zf[c + k] *= zscale;
            }
        }
        pend = kWaiting | (c_nh == n_nh - 1 ? kLastPass : 0) | (c_bg == 0 ? kFirstBg : 0) |
               (c_bg == a.n_bg - 1 ? kLastBg : 0) | (slow ? kSlow : 0);
        pend_x = x_row;
        pend_tile = c_t;
    }
    // The row sums of the pass before may still be read by a slow warp: a pass is
    // finished only after a barrier that follows the finish of the one before.
    __syncthreads();
    if (!failed) finish_pending();
    if (__syncthreads_or(failed ? 1 : 0)) {
        // a wait ran out (bounded): no value of this CTA's tiles is vouched for
        if (own_row)
            for (int i = t_begin; i < t_end; ++i)
                reinterpret_cast<T *>(a.v)[(long long)i * ROWS + tid] = (T)__longlong_as_double(0x7ff8000000000000ll);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

template <bool F64>
static tt_fsi_status launch(Args a, cudaStream_t st) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(masked_game_split_kernel<F64>, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<F64>::BYTES);
    if (e != cudaSuccess) return TT_FSI_ERR_CUDA;
    a.halves = 2 * a.n_tiles <= sms;
    const unsigned grid = (unsigned)(a.halves ? 2 * a.n_tiles : std::min<long long>(a.n_tiles, sms));
    masked_game_split_kernel<F64><<<grid, THREADS, Smem<F64>::BYTES, st>>>(a);
    e = cudaGetLastError();
    if (e == cudaSuccess) return TT_FSI_OK;
    return e == cudaErrorMemoryAllocation ? TT_FSI_ERR_NO_MEMORY : TT_FSI_ERR_CUDA;
}

// Narrower models stay on masked_game_kernel: a tile costs this path 7 us
// (float64) or 4 us (float32) of one SM whatever its width (16 instances, d = 14,
// float64: 2 x 2 units 131 us there and 116 to 182 here, by how many instances fit,
// 4 x 4 235 and 116; float32, 24 x 24: 60.5 and 61), and in float64 the prologue of
// a few tiles costs more than 4 x 4 units do (one instance, d = 7: 25 and 28).
bool split_serves(int d, int h1, int h2, long long B, int out_f32) {
    if (d < LOW || h1 > MAXH || h2 > MAXH) return false;
    if (out_f32) return h1 * h2 >= 26 * 26;
    return h1 + h2 >= ((B << (d - LOW)) >= 152 ? 8 : 12);
}

tt_fsi_status split_launch(const tt_fsi_mlp *model, const double *x_dev, const double *bg_dev, int n_bg, long long B,
                           void *v_dev, int out_f32, struct CUstream_st *stream) {
    Args a{};
    a.W1 = model->W1;
    a.b1 = model->b1;
    a.W2 = model->W2;
    a.b2 = model->b2;
    a.W3 = model->W3;
    a.b3 = model->b3;
    a.W2f = model->W2f;
    a.b2f = model->b2f;
    a.W3f = model->W3f;
    a.x = x_dev;
    a.bg = bg_dev;
    a.v = v_dev;
    a.n_bg = n_bg;
    a.d = model->d;
    a.h1 = model->h1;
    a.h2 = model->h2;
    a.n_tiles = B << (model->d - LOW);
    a.halves = 0;
    a.scale = 1.0 / (double)n_bg;
    a.two = 2;
    for (int k = 0; k < 4; ++k) a.unit[k] = 1 << (24 - 8 * k);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    return out_f32 ? launch<false>(a, st) : launch<true>(a, st);
}

}  // namespace ttfsi_mgs
