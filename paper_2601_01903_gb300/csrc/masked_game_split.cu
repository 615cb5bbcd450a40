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
//     to fixed point against a power-of-two scale and written as balanced
//     base-256 digits (float64: 7 digits = 56 bits, float32: 4 = 32 bits), each
//     an exact FP16 number.  A product of two digit matrices over K <= 128 has
//     sums below 2^21, so all products of one diagonal i + j = const add up
//     exactly in one FP32 accumulator (at most 7 of them, below 2^24): the
//     Ozaki splitting (Ozaki, Ogita, Oishi & Rump, "Error-free transformations
//     of matrix multiplication", 2012) with fixed digits.  Diagonals 0 .. 7
//     (float64, 34 products) or 0 .. 3 (float32, 10) are kept: what is dropped
//     is below the rounding of the last digit.  The diagonals are put together
//     in 64-bit integers (float64) or by three fused multiply-adds (float32).
//   float64 everywhere else is 64-bit fixed point on the integer pipes, which
//     are some 60 times as wide as the float64 pipe of this part: layer-1
//     pre-activations are sums of integers (exact, by subset sums), GELU is
//     max(z, 0) - |z| Phi(-|z|) with the second term from a table of quintic
//     polynomials, layer 3 exact 32 x 32-bit products.
//
// One CTA (16 warps) per SM walks a contiguous range of 128-coalition tiles:
// layer 1 of a tile into the digit slices in shared memory, one thread issues
// its MMAs, and while they run all warps do layers 2 (GELU) and 3 of the tile
// before, whose accumulators they drained into registers.
//
// Measured on one GB300: float64, 64 instances of a 14-64-64-1 model (2^20
// coalitions) 19.67 ms on masked_game_kernel, 0.79 ms here; float32, 8
// instances of a 16-128-128-1 model (2^19) 2.38 ms, 0.255 ms here.  Errors
// against 120-bit arithmetic are below masked_game_kernel's (relative 2-norms
// 0.7 to 3e-16 against 0.9 to 5e-16, and 1.1 to 1.9e-7 against 1 to 2.5e-7).
// Bound: instruction issue of the GELUs (float64: 112 instructions per hidden
// unit and coalition, 45 % issue; the tensor cores are 14 % busy).
//
// Instances (or background rows) whose scale the fixed point does not serve --
// non-finite values, one feature outweighing all others 256 to 1, in float64
// pre-activations that all stay below 1/4 or pass 2^16 -- are evaluated by
// slow_tile in the arithmetic of the type, tile by tile.
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
};

// ---- GELU in fixed point ---------------------------------------------------
// |z| Phi(-|z|) on intervals of width 2^-7, |z| < 8.75 (beyond it is below
// 2^-56 and taken as 0): per interval the quintic in tau = 256 (|z| - centre)
// that remains of its Taylor polynomial of degree 7 when the two highest
// Chebyshev terms are dropped, coefficients rounded to fixed point from the
// highest down: c0 (62 fraction bits), c1 (71), c2 (80; its low 16 bits hold
// c5), c3 (57), c4 (58), c5 (59).  Largest error against 160-bit arithmetic
// 2^-56.9, root mean square 2^-59.4 (float64's own rounding of a result near
// 1/3 is up to 2^-55).
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

// GELU of z = Z 2^-f as an integer of the same format, 43 <= f <= 62.  What
// bounds it is the integer ALU (half the issue rate), so shifts and adds are
// left to multiplications where the formats allow it.
__device__ __forceinline__ i64 gelu_fixed(i64 Z, int f, const ulonglong2 *tab, int two) {
    const int sign = hi32(Z) >> 31;
    const i64 m = (Z ^ join((unsigned)sign, sign)) - (i64)sign;
    const unsigned mh = (unsigned)hi32(m);
    const unsigned idx = min(mh >> (f - 39), (unsigned)TAB_INTERVALS);
    // tau 2^63: the bits below the index, about the centre
    const int t = (int)(__funnelshift_l(lo32(m), mh, 71 - f) ^ 0x80000000u);
    const unsigned tlow = lo32(m) << (71 - f);
    const ulonglong2 r0 = tab[2 * idx], r1 = tab[2 * idx + 1];
    const int u4 = (int)(r1.y >> 32) + __mulhi(t, (int)(short)(r1.x & 0xffff));
    const int u3 = (int)(unsigned)r1.y + __mulhi(t, u4);
    const int th = t >> 8, tl = (int)(__funnelshift_r(tlow, (unsigned)t, 8) >> 1);  // tau 2^55
    const i64 u2 = mad_wide(th, u3, mad_wide(__mulhi(tl, u3), two, (i64)r1.x));
    const i64 u1 = mul_hi_add(th, tl, u2, (i64)r0.y, two);
    const i64 h = mul_hi_add(th, tl, u1, (i64)r0.x, two);  // near z = 0 possibly a unit below 0
    return (Z & ~join((unsigned)sign, sign)) - shr(h, 62 - f);
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
    static constexpr int A = 0;
    static constexpr int W = A + C::NS * SLICE_A;
    static constexpr int W_CHUNKS = F64 ? 1 : 2;  // K chunks of W2 held (float32: all of it)
    static constexpr int TAB = W + W_CHUNKS * C::NS * C::NW * 128;
    static constexpr int PH = TAB + (F64 ? TAB_ROWS * 32 : 0);  // [16][KC] pre-activations by bits 3 .. 6
    static constexpr int DL = PH + 16 * KC * 8;                 // [7][KC] i64, or two chunks of [7][KC] int
    static constexpr int PART = DL + LOW * KC * 8;              // [3][ROWS] row sums of column groups 1 .. 3
    static constexpr int N8A = PART + 3 * ROWS * (F64 ? 16 : 4);              // [NW] 8 bytes: b2 in fixed point | b2, W3
    static constexpr int N8B = N8A + C::NW * 8;                 // [NW] int2: W3 in fixed point, high and low part
    static constexpr int L1 = N8B + C::NW * 8;                  // [MAXH] float: row sums of |W2|
    static constexpr int END = L1 + MAXH * 4;
    static constexpr int BYTES = END + 1024;
};
static_assert(Smem<true>::BYTES <= 232448 - 1024 && Smem<false>::BYTES <= 232448 - 1024, "fits one CTA per SM");

// Largest (op > 0) or smallest value over the CTA; every thread gets it.
__device__ __forceinline__ int block_max(int v, int *red) {
    v = __reduce_max_sync(0xffffffffu, v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    int m = red[0];
#pragma unroll
    for (int w = 1; w < WARPS; ++w) m = max(m, red[w]);
    return m;
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

// One tile of one background row in the arithmetic of the type (64 coalitions
// at a time; eight threads share a coalition's layer 2): thread c < 128
// returns f of coalition c.
template <typename T>
__device__ __noinline__ T slow_tile(const Args &a, const double *x, const double *base, long long S_high,
                                    unsigned char *smem) {
    T *pre = reinterpret_cast<T *>(smem);
    T *part = pre + 64 * (MAXH + 1);
    const int tid = threadIdx.x, ld = a.h1 + 1;
    T result = 0;
    for (int half = 0; half < 2; ++half) {
        const long long S0 = S_high | (half << 6);
        for (int j = tid; j < a.h1; j += THREADS) {
            double acc = a.b1[j];
            for (int i = 0; i < a.d; ++i) {
                const bool on = i >= 6 && ((S0 >> i) & 1);
                acc += a.W1[(long long)j * a.d + i] * (on ? x[i] : base[i]);
            }
            pre[j] = (T)acc;
            for (int k = 0; k < 6; ++k) {
                const T delta = (T)(a.W1[(long long)j * a.d + k] * (x[k] - base[k]));
                for (int c = 0; c < (1 << k); ++c) pre[(c | (1 << k)) * ld + j] = pre[c * ld + j] + delta;
            }
        }
        __syncthreads();
        for (int idx = tid; idx < 64 * a.h1; idx += THREADS) {
            const int c = idx / a.h1, j = idx - c * a.h1;
            pre[c * ld + j] = gelu_of(pre[c * ld + j]);
        }
        __syncthreads();
        const int c = tid & 63, q = tid >> 6;
        T acc3 = 0;
        for (int n = q; n < a.h2; n += 8) {
            T acc = Weights<T>::b2(a)[n];
            const T *w = Weights<T>::w2(a) + (long long)n * a.h1;
            for (int i = 0; i < a.h1; ++i) acc += __ldg(w + i) * pre[c * ld + i];
            acc3 += Weights<T>::w3(a)[n] * gelu_of(acc);
        }
        part[tid] = acc3;
        __syncthreads();
        if ((tid >> 6) == half) {
            T s = part[c];
            for (int k = 1; k < 8; ++k) s += part[c + 64 * k];
            result = s + (T)a.b3;
        }
        __syncthreads();
    }
    return result;
}

template <bool F64>
__global__ void __launch_bounds__(THREADS, 1) masked_game_split_kernel(const __grid_constant__ Args a) {
    using C = Cfg<F64>;
    using S = Smem<F64>;
    using T = typename std::conditional<F64, double, float>::type;
    constexpr int NS = C::NS, ND = C::ND, NW = C::NW, BITS = C::BITS, CPT = C::CPT;
    extern __shared__ __align__(1024) unsigned char sm_raw[];
    const uint32_t raw = smem_u32(sm_raw);
    unsigned char *sm = sm_raw + (((raw + 1023) & ~1023u) - raw);
    unsigned char *smA = sm + S::A, *smW = sm + S::W;
    ulonglong2 *tab = reinterpret_cast<ulonglong2 *>(sm + S::TAB);
    // layer-1 pre-activations: 62 (float64) or 30 (float32) fraction bits of 2^E
    using P = typename std::conditional<F64, i64, int>::type;
    constexpr int PBITS = F64 ? 62 : 30;
    constexpr int CHUNKS = F64 ? 1 : 2;  // K chunks whose tables are kept
    P *PH = reinterpret_cast<P *>(sm + S::PH);
    P *DL = reinterpret_cast<P *>(sm + S::DL);
    float *sL1 = reinterpret_cast<float *>(sm + S::L1);
    __shared__ __align__(8) uint64_t mbar, ph_ready, part_ready;  // MMAs done; tables made; row sums written
    __shared__ uint32_t tmem_sh;
    __shared__ int red[WARPS];

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
    }
    if constexpr (F64)
        for (int i = tid; i < TAB_ROWS * 2; i += THREADS) tab[i] = (&g_gelu_table[0][0])[i];

    // ---- once per CTA: the scale of W2 (2^ew), its row sums, the scale of W3 ----
    int ew, e3;
    bool model_ok;
    float ab2 = 0.f;  // |b2| of unit tid >> 2
    {
        const int n = tid >> 2, q = tid & 3;
        float mx = 0.f, sum = 0.f, aw3 = 0.f;
        if (n < a.h2) {
            for (int j = q; j < a.h1; j += 4) {
                const float w = fabsf((float)a.W2[(long long)n * a.h1 + j]);
                mx = fmaxf(mx, w);
                sum += w;  // carries a NaN or an infinity on
            }
            ab2 = fabsf((float)a.b2[n]);
            aw3 = fabsf((float)a.W3[n]);
        }
        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
        sum += __shfl_xor_sync(0xffffffffu, sum, 2);
        if (q == 0) sL1[n] = sum;
        ew = block_max(exp_above(1.01f * mx), red);
        e3 = block_max(exp_above(aw3), red);
        const bool bad = !(sum < 1e20f) || !(ab2 < 1e20f) || !(aw3 < 1e20f);
        model_ok = block_max(bad ? 1 : 0, red) == 0 && e3 < 60;
        ew = max(ew, -60);  // an all-zero W2 has any scale
        e3 = max(e3, -60);
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_sh;
    const uint32_t a_base = smem_u32(smA), w_base = smem_u32(smW);  // below 2^18: descriptors add up

    const int n_kc = (a.h1 + KC - 1) / KC, n_nh = (a.h2 + NW - 1) / NW;
    const int tile_shift = a.d - LOW;
    const long long t_begin = a.n_tiles * blockIdx.x / gridDim.x, t_end = a.n_tiles * (blockIdx.x + 1) / gridDim.x;
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

    // epilogue state: the accumulators of the pass in flight, its row sums so
    // far, and (threads < 128) the sum over background rows of row tid
    i64 zi[F64 ? CPT : 1];
    float zf[F64 ? 1 : CPT];
    i64 acc_hh = 0, acc_hl = 0, acc_lh = 0, acc_ll = 0;
    float acc_f = 0.f;
    T vsum = 0;
    bool pending = false, pend_last_nh = false, pend_first_bg = false, pend_last_bg = false;
    int pend_f2 = 0;
    long long pend_tile = 0;

    // epilogue: thread (row, quarter of the pass's columns), in whole loads of 8
    const int n_col = min(NW, a.h2);
    const int cpt = min(CPT, ((n_col + 31) >> 5) << 3);
    const int erow = 32 * (warp & 3) + lane, ecol = (warp >> 2) * cpt;

    auto emit = [&](T f, bool first, bool last, long long tile) {  // threads < 128
        if (a.n_bg == 1)
            vsum = f;
        else
            vsum = first ? (T)a.scale * f : vsum + (T)a.scale * f;
        if (last) reinterpret_cast<T *>(a.v)[tile * ROWS + tid] = vsum;
    };

    // Layers 2 (GELU) and 3 of the drained accumulators.
    auto finish_pending = [&]() {
        if (!pending) return;
        pending = false;
        if constexpr (F64) {
            const i64 *b2q = reinterpret_cast<const i64 *>(sm + S::N8A) + ecol;
            const int2 *w3q = reinterpret_cast<const int2 *>(sm + S::N8B) + ecol;
            // eight columns an iteration from the front of the register array,
            // which then moves up (a run-time loop keeps the code short)
#pragma unroll 1
            for (int c = 0; c < cpt; c += 8) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const i64 g = gelu_fixed(zi[k] + b2q[c + k], pend_f2, tab, a.two);
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
            const float2 *p2 = reinterpret_cast<const float2 *>(sm + S::N8A) + ecol;
#pragma unroll 1
            for (int c = 0; c < cpt; c += 8) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float2 p = p2[c + k];  // b2, W3
                    acc_f = fmaf(p.y, gelu_fast(zf[k] + p.x), acc_f);
                }
#pragma unroll
                for (int k = 0; k + 8 < CPT; ++k) zf[k] = zf[k + 8];
            }
        }
        if (pend_last_nh) {
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
                    // units 2^-(f2 + 53 - e3), and 2^(65 - lz) of them (2 when all is in the low word)
                    const int e = 65 - lz - (pend_f2 + 53 - e3);
                    emit(s * __longlong_as_double((i64)(1023 + e) << 52) + a.b3, pend_first_bg, pend_last_bg, pend_tile);
                }
            } else {
                float *pf = reinterpret_cast<float *>(sm + S::PART);
                if (group) {
                    pf[(group - 1) * ROWS + erow] = acc_f;
                    arrive(&part_ready);
                } else {
                    wait(&part_ready, part_parity);
                    const float s = (acc_f + pf[tid]) + (pf[ROWS + tid] + pf[2 * ROWS + tid]);
                    emit(s + (float)a.b3, pend_first_bg, pend_last_bg, pend_tile);
                }
            }
            acc_hh = acc_hl = acc_lh = acc_ll = 0;
            acc_f = 0.f;
        }
    };

    // ---- the walk over (tile, background row, pass over layer 2, K chunk) ----
    long long t = t_begin;
    int bgi = 0, nh = 0, kc = 0;
    long long key = -1;        // (instance, background row) the scales were made for
    long long const_key = -1;  // key and nh of the epilogue's per-unit constants
    int chunk_key = -1;        // last chunk (of key) that DL, dhigh and base0 were made for
    int w_key = -1;            // (nh, kc) of the resident slices of W2 (float32: the chunks made)
    int E = 0, f2 = 0;         // layer 1 stays below 2^E; fraction bits of layer 2 (float64)
    bool ok = false;
    P dhigh[CHUNKS][3] = {}, base0[CHUNKS] = {};
    // layer-1 tables: lanes 8 v + part of a warp have unit 4 warp + v of the chunk
    const int part = lane & 7, jj = 4 * warp + (lane >> 3);

    // The layer-1 tables of the step at (t, bgi, kc), after every warp is done
    // with those before: scales when the instance or background row changes,
    // then PH[e][j] = the empty coalition's pre-activation + the high features'
    // + those of bits 3 .. 6 (pattern e).
    auto prepare_step = [&]() {
        const long long inst = t >> tile_shift;
        const long long S_high = (t - (inst << tile_shift)) << LOW;
        const double *x = a.x + inst * a.d;
        const double *base = a.bg + (long long)bgi * a.d;
        if (key != inst * a.n_bg + bgi) {
            key = inst * a.n_bg + bgi;
            chunk_key = -1;
            const int j = tid >> 2, q = tid & 3;
            float bound = 0.f, top = 0.f;
            if (j < a.h1) {
                for (int i = q; i < a.d; i += 4) {
                    const float xi = (float)x[i], zi0 = (float)base[i];
                    // (a NaN or an infinity of either carries through the second term)
                    const float m = fmaxf(fabsf(xi), fabsf(zi0)) + 0.f * (xi + zi0);
                    const float c = fabsf((float)a.W1[(long long)j * a.d + i]) * m;
                    bound += c;
                    top = fmaxf(top, c);
                }
                if (q == 0) bound += fabsf((float)a.b1[j]);
            }
            for (int o = 1; o < 4; o <<= 1) {
                bound += __shfl_xor_sync(0xffffffffu, bound, o);
                top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
            }
            const bool finite = bound < 1e20f;
            const int e = finite ? exp_above(1.01f * bound) : 100;
            E = block_max(e, red);
            const bool lone = finite && e >= E - 2 && e > -100 && (bound - top) < 0.00390625f * top;
            ok = model_ok && block_max(lone ? 1 : 0, red) == 0;
            if constexpr (F64) {
                ok = ok && E >= -1 && E <= 16;
                E = max(E, 0);
                // pre-activations of layer 2 stay below 2^ze
                const float zb = ok ? 1.02f * pow2(E) * sL1[j] + ab2 : 0.f;
                const int ze = block_max(exp_above(zb), red);
                f2 = min(62, 61 - ze);
                // (its accumulators come in units of 2^(E + ew - 55))
                ok = ok && ze <= 18 && ze >= -5 && E + ew + f2 >= 40;
            } else {
                ok = ok && E > -50 && E < 60 && ew < 40;
            }
        }
        if (!ok) return;
        const int j = kc * KC + jj;
        const bool in = j < a.h1;
        const int slot = F64 ? 0 : kc;
        P *dl = DL + slot * (LOW * KC) + jj;
        if (F64 ? chunk_key != kc : chunk_key < kc) {
            // every feature's contribution when it joins the coalition: the low
            // seven in shared memory, the high ones (at most three per lane) in
            // registers; and the empty coalition's sum
            chunk_key = kc;
            const int f1 = PBITS - E;
            const double *w1 = a.W1 + (long long)(in ? j : 0) * a.d;
            P z0 = 0, dlow = 0, dh[3];
            if (in && part == 7) z0 = (P)fix(a.b1[j], f1);
            if (in && part < LOW) {
                z0 = (P)fix(w1[part] * base[part], f1);
                dlow = (P)fix(w1[part] * x[part], f1) - z0;
            }
            if (part < LOW) dl[part * KC] = dlow;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int i = LOW + part + 8 * k;
                dh[k] = 0;
                if (in && i < a.d) {
                    const P z = (P)fix(w1[i] * base[i], f1);
                    z0 += z;
                    dh[k] = (P)fix(w1[i] * x[i], f1) - z;
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
        P s = slot ? base0[CHUNKS - 1] : base0[0];
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if ((S_high >> (LOW + part + 8 * k)) & 1) s += slot ? dhigh[CHUNKS - 1][k] : dhigh[0][k];
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        // entries part and part + 8
#pragma unroll
        for (int m = 0; m < 3; ++m)
            if ((part >> m) & 1) s += dl[(3 + m) * KC];
        PH[part * KC + jj] = s;
        PH[(part + 8) * KC + jj] = s + dl[6 * KC];
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
        if (!ok) {
            if (__syncthreads_or(failed ? 1 : 0)) {
                failed = true;
                break;
            }
            finish_pending();  // (after a barrier: see the end of the walk)
            const long long inst = t >> tile_shift;
            const T f = slow_tile<T>(a, a.x + inst * a.d, a.bg + (long long)bgi * a.d, (t - (inst << tile_shift)) << LOW, smA);
            if (tid < ROWS) emit(f, bgi == 0, bgi == a.n_bg - 1, t);
            next_step();
            if (t < t_end) {
                prepare_step();
                arrive(&ph_ready);
            }
            continue;
        }
        // ---- layer 1: units 2u, 2u + 1 of the chunk; a warp has rows 8 warp ..
        // 8 warp + 7, split over its lanes when the chunk has at most 32 or 16
        // units; a lane walks its rows in pairs (bit 0), the pairs in Gray-code order ----
        {
            const int units = min(KC, a.h1 - kc * KC);
            const int lg = units <= 16 ? 3 : units <= 32 ? 4 : 5, nb = lg - 2;
            const int u = lane & ((1 << lg) - 1), sub = lane >> lg;
            const P *ph = PH + warp * KC + 2 * u, *dl = DL + (F64 ? 0 : kc * (LOW * KC)) + 2 * u;
            P pa = ph[0], pb = ph[1], da[3], db[3];
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                da[m] = dl[m * KC];
                db[m] = dl[m * KC + 1];
                if (m >= nb && ((sub >> (m - nb)) & 1)) {
                    pa += da[m];
                    pb += db[m];
                }
            }
            const int row0 = 8 * warp + (sub << nb);
            const float down = F64 ? 0.f : pow2(E - 30), up = F64 ? 0.f : pow2(31 - E);
            auto put = [&](P za, P zb, int row) {
                unsigned char *dst = smA + pair_offset(row, u);
                if constexpr (F64) {
                    // rounded to 55 fraction bits and biased
                    const u64 c = (BIAS7 << 7) + 64;
                    put_digits(dst, SLICE_A, ((u64)gelu_fixed(za, 62 - E, tab, a.two) + c) >> 7,
                               ((u64)gelu_fixed(zb, 62 - E, tab, a.two) + c) >> 7);
                } else {
                    put_digits(dst, SLICE_A, (unsigned)__float2int_rn(gelu_fast((float)za * down) * up) + BIAS4,
                               (unsigned)__float2int_rn(gelu_fast((float)zb * down) * up) + BIAS4);
                }
            };
#pragma unroll 1
            for (int q = 0; q < (1 << (nb - 1)); ++q) {
                if (q == 1) {
                    pa += da[1];
                    pb += db[1];
                } else if (q == 2) {
                    pa += da[2];
                    pb += db[2];
                } else if (q == 3) {
                    pa -= da[1];
                    pb -= db[1];
                }
                const int row = row0 + 2 * (q ^ (q >> 1));
                put(pa, pb, row);
                put(pa + da[0], pb + db[0], row + 1);
            }
        }
        // ---- the slices of W2 for (nh, kc) (float64: one chunk is held;
        // float32: both, made with the first tile) ----
        if (F64 ? w_key != nh * n_kc + kc : w_key < kc) {
            w_key = F64 ? nh * n_kc + kc : kc;
            unsigned char *w_dst = smW + (F64 ? 0 : kc * (NS * NW * 128));
            const int u = lane, j0 = kc * KC + 2 * u;
            for (int n = warp; n < NW; n += WARPS) {
                const int gn = nh * NW + n;
                i64 wa = 0, wb = 0;
                if (gn < a.h2) {
                    const double *w = a.W2 + (long long)gn * a.h1;
                    if (j0 < a.h1) wa = fix(w[j0], BITS - ew);
                    if (j0 + 1 < a.h1) wb = fix(w[j0 + 1], BITS - ew);
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
        const int c_nh = nh, c_bg = bgi, c_E = E, c_f2 = f2;
        const long long c_t = t, c_key = key;
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
        if (last_kc && const_key != c_key * n_nh + c_nh) {
            // per-unit constants of this pass's epilogue
            const_key = c_key * n_nh + c_nh;
            __syncthreads();
            if (tid < NW) {
                const int gn = c_nh * NW + tid;
                const bool in = gn < a.h2;
                if constexpr (F64) {
                    reinterpret_cast<i64 *>(sm + S::N8A)[tid] = in ? fix(a.b2[gn], c_f2) : 0;
                    const i64 w = in ? fix(a.W3[gn], 53 - e3) : 0;  // wh 2^27 + wl, |wl| <= 2^26
                    const int wh = (int)((w + (1ll << 26)) >> 27);
                    reinterpret_cast<int2 *>(sm + S::N8B)[tid] = make_int2(wh, (int)(w - ((i64)wh << 27)));
                } else {
                    reinterpret_cast<float2 *>(sm + S::N8A)[tid] =
                        in ? make_float2((float)a.b2[gn], (float)a.W3[gn]) : make_float2(0.f, 0.f);
                }
            }
            __syncthreads();
        }
        wait(&mbar, parity);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (!last_kc) continue;
        // ---- drain the accumulators of this pass into registers ----
        const int sl = F64 ? c_E + ew + c_f2 - 38 : 0;  // from units of 2^(E + ew - 38) to the format of layer 2
        const float zscale = F64 ? 0.f : pow2(c_E + ew - 14);
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
                // the parts are in units of 2^(E + ew - 38) and 2^(E + ew - 70)
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    zi[c + k] = join(lo32(up[k]) << sl, (int)__funnelshift_l(lo32(up[k]), (unsigned)hi32(up[k]), sl)) +
                                shr(low[k], 32 - sl);
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
        pending = true;
        pend_last_nh = c_nh == n_nh - 1;
        pend_first_bg = c_bg == 0;
        pend_last_bg = c_bg == a.n_bg - 1;
        pend_f2 = c_f2;
        pend_tile = c_t;
    }
    // The row sums of the pass before may still be read by a slow warp: a pass is
    // finished only after a barrier that follows the finish of the one before.
    __syncthreads();
    if (!failed) finish_pending();
    if (__syncthreads_or(failed ? 1 : 0)) {
        // a wait ran out (bounded): no value of this CTA's tiles is vouched for
        for (long long i = t_begin * ROWS + tid; i < t_end * ROWS; i += THREADS)
            reinterpret_cast<T *>(a.v)[i] = (T)__longlong_as_double(0x7ff8000000000000ll);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

template <bool F64>
static tt_fsi_status launch(const Args &a, cudaStream_t st) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(masked_game_split_kernel<F64>, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<F64>::BYTES);
    if (e != cudaSuccess) return TT_FSI_ERR_CUDA;
    const unsigned grid = (unsigned)std::min<long long>(a.n_tiles, sms);
    masked_game_split_kernel<F64><<<grid, THREADS, Smem<F64>::BYTES, st>>>(a);
    e = cudaGetLastError();
    if (e == cudaSuccess) return TT_FSI_OK;
    return e == cudaErrorMemoryAllocation ? TT_FSI_ERR_NO_MEMORY : TT_FSI_ERR_CUDA;
}

// Float32 models of fewer than 24 x 24 hidden units stay on masked_game_kernel:
// a tile costs this path about 4 us of one SM whatever its width.
bool split_serves(int d, int h1, int h2, int out_f32) {
    return d >= LOW && h1 <= MAXH && h2 <= MAXH && (!out_f32 || h1 * h2 >= 24 * 24);
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
    a.scale = 1.0 / (double)n_bg;
    a.two = 2;
    for (int k = 0; k < 4; ++k) a.unit[k] = 1 << (24 - 8 * k);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    return out_f32 ? launch<false>(a, st) : launch<true>(a, st);
}

}  // namespace ttfsi_mgs
