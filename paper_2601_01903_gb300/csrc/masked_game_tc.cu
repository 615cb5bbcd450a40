// Masked-model value function on the tcgen05 tensor cores (label path).
//
// v_x(S) = f(z), z_i = x_i for i in S and baseline_i otherwise, f the GELU
// MLP d -> 128 -> 128 -> 1 (Section 2.1's value function of a model with
// absent features set to a baseline).  One CTA (8 warps) takes 128
// coalitions at a time:
//   layer 1 (CUDA cores): a thread owns two neighbouring hidden units, held as
//     one packed FP32 pair, and 32 coalitions.  For the consecutive coalitions
//     of a dense tile it walks their 5 low bits in Gray-code order (one packed
//     add per coalition, every flip a compile-time constant); for a list of
//     coalitions it forms the d-term dot products, 8 rows at a time -- then
//     GELU, rounded to BF16 into shared memory in the 128-byte-swizzled
//     K-major layout the tensor cores read;
//   layer 2 (tensor cores): eight tcgen05.mma (M = 128 coalitions, N = 128
//     units, K = 16 each) of the BF16 activations against W2 (rounded to BF16
//     once per CTA and kept in shared memory), FP32 accumulators in tensor
//     memory, completion signalled on an mbarrier (bounded wait);
//   layer 3 (epilogue): warps w and w + 4 read accumulator rows 32w..32w+31
//     (their TMEM lane quarter), columns 0-63 and 64-127, with tcgen05.ld and
//     form b3 + sum_n W3[n] GELU(acc[n] + b2[n]) in FP32, pairs of columns
//     packed.
// The interventional value function of Section 4.1 (the mean of f over
// background rows standing in for the absent features) repeats the three
// layers per background row on the same tile and averages in FP32; one row
// is the baseline value function.  When the tiles alone do not fill the GPU, a
// cluster of CTAs shares a tile's rows and adds its sums in rank order through
// distributed shared memory.  The BF16 rounding of the layer-2 operands is this
// path's precision (masked_game_split.cu is the parity path).
//
// What bounds it is the 256 GELUs of a coalition on the FP32 pipe (packed
// FP32 instructions halve the issue slots, not the pipe's time) with the
// special-function unit close behind; three CTAs per SM run one another's
// phases, and one barrier per pass is left.  Layer 1 keeps its formula and the
// order of its sums: a last-bit change there flips roundings to BF16, which
// the outputs see.  One GB300, d = 16, 64 instances, one baseline: 1.75 ms at
// two CTAs per SM (an occupancy query said one) with scalar arithmetic and float64
// conversions in every thread, 0.70 ms now; d = 12, 8 instances, 100 rows: 1.07 ms and
// 0.70 ms (clusters of 5 share the rows of 256 tiles).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

// only the tcgen05 helpers (the GEMM kernel itself lives in student.cu)
#define TTFSI_GEMM_HELPERS_ONLY
#include "gemm_tcgen05.cuh"
#include "tt_fsi.h"

namespace ttfsi_mgtc {

using ttfsi_gemm::mbar_init;
using ttfsi_gemm::mbar_wait;
using ttfsi_gemm::mma_bf16;
using ttfsi_gemm::mma_commit;
using ttfsi_gemm::smem_desc;
using ttfsi_gemm::smem_u32;

constexpr int ROWS = 128;                  // coalitions per tile (MMA M)
constexpr int H = 128;                     // hidden width (MMA N and K)
constexpr int THREADS = 256;  // 8 warps
constexpr int KB_BYTES = ROWS * 128;       // one 64-wide K block of 128 rows: 16 KB
constexpr int OPERAND_BYTES = 2 * KB_BYTES;  // K = 128: two blocks
constexpr int kErrTimeout = 1;
constexpr int MAX_CLUSTER = 8;
constexpr int LIST_INST = 6;  // instances a tile of listed rows can span when K >= 32

struct Args {
    const float *W1, *b1, *W2, *b2, *W3;
    float b3;
    const double *x, *base;  // base: n_bg background rows [n_bg, d] (one row: the baseline)
    int n_bg;
    int d;
    const unsigned *coal;  // list mode: rows are (instance r / K, coal[r])
    int K;
    float *out;
    long long n_tiles, n_rows;
    int *err;
};

// Shared memory: the two operands, W1 transposed (dense mode: at most 16 rows,
// which leaves room for three CTAs per SM; the other features' weights come
// through L1), and in list mode the tile's input vectors [d][ROWS], each value
// twice (a packed pair).
constexpr int W1_ROWS = 16;
__host__ __device__ constexpr int w1_rows(int d, bool list) { return list || d < W1_ROWS ? d : W1_ROWS; }
__host__ __device__ constexpr int smem_bytes(int d, bool list) {
    return 2 * OPERAND_BYTES + w1_rows(d, list) * H * 4 + (list ? d * ROWS * 8 : 0);
}

// ---- packed FP32 pairs --------------------------------------------------------
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack(f2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 both(float c) { return pack(c, c); }
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// GELU of a pair, layer 1: z Phi(z) with the normal tail by Abramowitz &
// Stegun, Handbook of Mathematical Functions, formula 7.1.26 (Hastings'
// approximation of erfc(x) = P(t) exp(-x^2), t = 1 / (1 + p x), x >= 0;
// absolute error of erf below 1.5e-7, far below the BF16 rounding that
// follows): Phi(z) = 1 - q for z >= 0 and q for z < 0, q = erfc(|z| / sqrt 2) / 2
// (P halved).
__device__ __forceinline__ f2 gelu_layer1(f2 z) {
    float z0, z1;
    unpack(z, z0, z1);
    const f2 az = z & 0x7fffffff7fffffffull;
    const f2 x = mul2(az, both(0.70710678118654752f));
    float u0, u1;
    unpack(fma2(both(0.3275911f), x, both(1.0f)), u0, u1);
    const f2 t = pack(rcp_approx(u0), rcp_approx(u1));
    f2 p = fma2(both(0.5f * 1.061405429f), t, both(0.5f * -1.453152027f));
    p = fma2(p, t, both(0.5f * 1.421413741f));
    p = fma2(p, t, both(0.5f * -0.284496736f));
    p = fma2(p, t, both(0.5f * 0.254829592f));
    float y0, y1;
    unpack(mul2(mul2(x, x), both(-1.4426950408889634f)), y0, y1);
    const f2 q = mul2(mul2(p, t), pack(ex2_approx(y0), ex2_approx(y1)));
    float q0, q1, c0, c1;
    unpack(q, q0, q1);
    unpack(fma2(q, both(-1.0f), both(1.0f)), c0, c1);
    return mul2(z, pack(z0 >= 0.f ? c0 : q0, z1 >= 0.f ? c1 : q1));
}

// k GELU(z) of a pair, layer 3, from y = k z, k = sqrt(log2(e) / 2) (so that
// exp(-z^2 / 2) = 2^(-y^2)): max(y, 0) - t exp(-z^2 / 2) Q, t = |y|, Q = k
// exp(z^2 / 2) Phi(-|z|) / t as s P(s), s = 1 / (1 + 0.28 |z|), P of degree 5
// (weighted least squares, refitted to an even error; that of the result is
// 3.4e-9, below the rounding of FP32).  An infinite y gives max(y, 0), a NaN NaN.
constexpr float L3_SCALE = 0.84932180028801907f;  // k
__device__ __forceinline__ f2 gelu_layer3(f2 y) {
    float y0, y1, t0, t1;
    unpack(y, y0, y1);
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(t0) : "f"(fabsf(y0)), "f"(1e30f));
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(t1) : "f"(fabsf(y1)), "f"(1e30f));
    const f2 t = pack(t0, t1);
    float u0, u1, e0, e1;
    unpack(fma2(both(0.28f / L3_SCALE), t, both(1.0f)), u0, u1);
    unpack(mul2(mul2(t, both(-1.0f)), t), e0, e1);
    const f2 s = pack(rcp_approx(u0), rcp_approx(u1));
    f2 p = fma2(both(0.10755508235538286f), s, both(-0.39699074731224754f));  // -P
    p = fma2(p, s, both(0.24851913789490362f));
    p = fma2(p, s, both(-0.27818327722545133f));
    p = fma2(p, s, both(-0.06379108976018237f));
    p = fma2(p, s, both(-0.11710905724886507f));
    const f2 q = mul2(mul2(t, s), pack(ex2_approx(e0), ex2_approx(e1)));
    return fma2(q, p, pack(fmaxf(y0, 0.f), fmaxf(y1, 0.f)));
}

// Byte offset of element (row r, column k) of a 128 x 128 BF16 operand in
// two 128-byte-swizzled K blocks.
__device__ __forceinline__ uint32_t operand_offset(int r, int k) {
    return (uint32_t)((k >> 6) * KB_BYTES + r * 128 + ((((k & 63) >> 3) ^ (r & 7)) << 4) + (k & 7) * 2);
}

__device__ __forceinline__ void store_pair(unsigned char *dst, f2 v) {
    float a, b;
    unpack(v, a, b);
    *reinterpret_cast<__nv_bfloat162 *>(dst) = __floats2bfloat162_rn(a, b);
}

template <bool LIST>
__global__ void __launch_bounds__(THREADS, LIST ? 2 : 3) masked_game_tc_kernel(const __grid_constant__ Args a) {
    extern __shared__ __align__(1024) unsigned char sm_raw[];
    unsigned char *wB = sm_raw;                  // W2 as the B operand [n][k]
    unsigned char *aA = wB + OPERAND_BYTES;      // activations as the A operand [row][k]
    float *w1t = reinterpret_cast<float *>(aA + OPERAND_BYTES);  // [w1_rows][H]
    f2 *zT = reinterpret_cast<f2 *>(w1t + w1_rows(a.d, LIST) * H);  // list mode: [d][ROWS]
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base_sh;
    __shared__ __align__(16) float sb2[H], sw3[H];
    __shared__ float2 sxb[2][32];                // the pass's features and background row, float32; double-buffered
    __shared__ float sx[LIST ? LIST_INST : 1][32];  // list mode: the features of the tile's instances
    __shared__ float spart[2][ROWS];             // the second column half's sums, by turns

    const int tid = threadIdx.x, warp = tid >> 5;
    if (smem_u32(sm_raw) & 1023u) {  // the swizzled operands need the declared alignment
        if (tid == 0) atomicOr(a.err, kErrTimeout);
        return;
    }
    uint32_t crank, csize;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(csize));
    if (tid < H) {
        sb2[tid] = a.b2[tid] * L3_SCALE;
        sw3[tid] = a.W3[tid] * (1.0f / L3_SCALE);
    }
    // W2 -> BF16 B operand, W1 transposed (once per CTA)
    for (int i = tid; i < H * H / 2; i += THREADS) {
        const int n = i / (H / 2), k = 2 * (i - n * (H / 2));
        *reinterpret_cast<__nv_bfloat162 *>(wB + operand_offset(n, k)) =
            __floats2bfloat162_rn(a.W2[n * H + k], a.W2[n * H + k + 1]);
    }
    for (int i = tid; i < w1_rows(a.d, LIST) * H; i += THREADS) w1t[i] = a.W1[(i & (H - 1)) * a.d + (i >> 7)];
    if (tid == 0) {
        mbar_init(smem_u32(&mbar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                     "r"(H));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }

    // units k0, k0 + 1 and rows 32 qr .. 32 qr + 31 of this thread's layer 1
    const int k0 = 2 * (tid & 63), qr = tid >> 6, row0 = qr << 5;
    const f2 bias1 = pack(a.b1[k0], a.b1[k0 + 1]);
    const int tile_shift = LIST ? 0 : a.d - 7;
    const int quarter = warp & 3, col0 = (warp >> 2) * (H / 2);
    const int bg0 = (int)((long long)a.n_bg * crank / csize), bg1 = (int)((long long)a.n_bg * (crank + 1) / csize);
    const long long t0 = blockIdx.x / csize, t_step = gridDim.x / csize;
    uint32_t parity = 0;
    int xbuf = 0, turn = 0;
    bool lost = false, failed = false;  // a wait of this thread's, of the CTA's, ran out
    float out_sum = 0.f;         // warps 0-3: the tile before's first-half sums, output pending
    long long out_tile = -1;

    // features (dense mode) and background row of a pass, as float32
    auto load_row = [&](long long t, int bgi) {
        const double *x = a.x + (LIST ? 0 : (t >> tile_shift) * a.d);
        return make_float2(LIST ? 0.f : (float)x[tid], (float)a.base[(long long)bgi * a.d + tid]);
    };
    auto write_out = [&](float sum, long long t) {  // warps 0-3
        const long long row = t * ROWS + tid;
        if (row < a.n_rows) a.out[row] = a.b3 + sum / (float)a.n_bg;
    };

    if (t0 < a.n_tiles && bg0 < bg1 && tid < a.d) sxb[0][tid] = load_row(t0, bg0);
    if (csize > 1)
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_sh;
    const uint32_t idesc = ttfsi_gemm::instr_desc_bf16(ROWS, H);
    const uint64_t da = smem_desc(smem_u32(aA)), db = smem_desc(smem_u32(wB));

    for (long long t = t0; t < a.n_tiles; t += t_step) {
        f2 vsum = 0;
        for (int bgi = bg0; bgi < bg1; ++bgi) {
            // the next pass's features and background row, on their way
            float2 next_xb = make_float2(0.f, 0.f);
            const bool more = bgi + 1 < bg1;
            if (tid < a.d && (more || t + t_step < a.n_tiles))
                next_xb = load_row(more ? t : t + t_step, more ? bgi + 1 : bg0);
            // ---- layer 1 into the A operand ----
            if constexpr (!LIST) {
                const unsigned cb = ((unsigned)(t & ((1ll << tile_shift) - 1)) << 7) | ((unsigned)qr << 5);
                f2 p = bias1, dl[5];
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    const float2 xb = sxb[xbuf][i];
                    const f2 w = *reinterpret_cast<const f2 *>(w1t + i * H + k0);
                    dl[i] = mul2(w, both(xb.x - xb.y));
                    p = fma2(w, both(xb.y), p);
                }
                for (int i = 5; i < min(a.d, W1_ROWS); ++i) {
                    const float2 xb = sxb[xbuf][i];
                    p = fma2(*reinterpret_cast<const f2 *>(w1t + i * H + k0), both(((cb >> i) & 1u) ? xb.x : xb.y), p);
                }
                for (int i = W1_ROWS; i < a.d; ++i) {
                    const float2 xb = sxb[xbuf][i];
                    p = fma2(pack(__ldg(a.W1 + k0 * a.d + i), __ldg(a.W1 + (k0 + 1) * a.d + i)),
                             both(((cb >> i) & 1u) ? xb.x : xb.y), p);
                }
#pragma unroll
                for (int r = 0; r < 32; ++r) {
                    if (r > 0) {
                        // the bit that flips between gray(r - 1) and gray(r), and its old value
                        const int q = (r & 1) ? 0 : (r & 2) ? 1 : (r & 4) ? 2 : (r & 8) ? 3 : 4;
                        const bool was_set = (((r - 1) ^ ((r - 1) >> 1)) >> q) & 1;
                        p = was_set ? fma2(dl[q], both(-1.0f), p) : add2(p, dl[q]);
                    }
                    store_pair(aA + operand_offset(row0 + (r ^ (r >> 1)), k0), gelu_layer1(p));
                }
            } else {
                // the rows' input vectors; with at least 32 rows per instance the
                // instances' features are converted once
                const long long first = t * ROWS;
                const long long inst0 = first / a.K;
                const bool staged = a.K >= 32;
                if (staged) {
                    const long long last = min(first + ROWS, a.n_rows) - 1;
                    const int n_inst = (int)(last / a.K - inst0) + 1;
                    for (int i = tid; i < n_inst * 32; i += THREADS)
                        if ((i & 31) < a.d) sx[i >> 5][i & 31] = (float)a.x[(inst0 + (i >> 5)) * a.d + (i & 31)];
                    __syncthreads();
                }
                {
                    const int r = tid & (ROWS - 1);
                    const long long row = first + r;
                    const bool in = row < a.n_rows;
                    const long long inst = in ? row / a.K : inst0;
                    const unsigned m = in ? a.coal[row] : 0u;
                    for (int i = tid >> 7; i < a.d; i += 2) {
                        float z = 0.f;
                        if (in) {
                            if ((m >> i) & 1u)
                                z = staged ? sx[inst - inst0][i] : (float)a.x[inst * a.d + i];
                            else
                                z = sxb[xbuf][i].y;
                        }
                        zT[i * ROWS + r] = both(z);
                    }
                }
                __syncthreads();
#pragma unroll 1
                for (int r0 = row0; r0 < row0 + 32; r0 += 8) {
                    f2 p[8];
#pragma unroll
                    for (int r = 0; r < 8; ++r) p[r] = bias1;
#pragma unroll 4
                    for (int i = 0; i < a.d; ++i) {
                        const f2 w = *reinterpret_cast<const f2 *>(w1t + i * H + k0);
                        const ulonglong2 *z = reinterpret_cast<const ulonglong2 *>(zT + i * ROWS + r0);
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const ulonglong2 zz = z[r];
                            p[2 * r] = fma2(w, zz.x, p[2 * r]);
                            p[2 * r + 1] = fma2(w, zz.y, p[2 * r + 1]);
                        }
                    }
#pragma unroll
                    for (int r = 0; r < 8; ++r) store_pair(aA + operand_offset(r0 + r, k0), gelu_layer1(p[r]));
                }
            }
            // ---- layer 2 on the tensor cores ----
            xbuf ^= 1;
            if (tid < a.d) sxb[xbuf][tid] = next_xb;
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            // A written, accumulators read, next features and the sums of the pass before in place
            failed = __syncthreads_or(lost ? 1 : 0) != 0;
            if (failed) break;
            if (tid == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int kb = 0; kb < 2; ++kb)
#pragma unroll
                    for (int k16 = 0; k16 < 4; ++k16)
                        mma_bf16(tmem, da + ((kb * KB_BYTES + k16 * 32) >> 4), db + ((kb * KB_BYTES + k16 * 32) >> 4), idesc,
                                 (kb > 0 || k16 > 0) ? 1u : 0u);
                mma_commit(smem_u32(&mbar));
            }
            // the output of the tile before, now that both halves' sums are in place
            if (warp < 4 && out_tile >= 0) write_out(out_sum + spart[turn ^ 1][tid], out_tile);
            out_tile = -1;
            lost |= !mbar_wait(smem_u32(&mbar), parity);  // every lane polls: the warp stays together
            parity ^= 1u;
            __syncwarp();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // ---- layer 3 in the epilogue: warps w, w + 4 share accumulator rows ----
#pragma unroll 1
            for (int c0 = col0; c0 < col0 + H / 2; c0 += 16) {
                uint32_t r[16];
                const uint32_t taddr = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)c0;
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
                    "[%16];"
                    : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                      "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                      "=r"(r[15])
                    : "r"(taddr));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int j = 0; j < 16; j += 4) {
                    const ulonglong2 b2 = *reinterpret_cast<const ulonglong2 *>(sb2 + c0 + j);
                    const ulonglong2 w3 = *reinterpret_cast<const ulonglong2 *>(sw3 + c0 + j);
                    vsum = fma2(w3.x, gelu_layer3(fma2(((f2)r[j + 1] << 32) | r[j], both(L3_SCALE), b2.x)), vsum);
                    vsum = fma2(w3.y, gelu_layer3(fma2(((f2)r[j + 3] << 32) | r[j + 2], both(L3_SCALE), b2.y)), vsum);
                }
            }
        }
        // ---- the tile's row sums ----
        float v0, v1;
        unpack(vsum, v0, v1);
        if (warp >= 4) spart[turn][tid - ROWS] = v0 + v1;
        if (csize == 1) {
            // written out during the next pass, after its barrier
            out_sum = v0 + v1;
            out_tile = t;
        } else {
            // through rank 0's activations, once every rank is done with the tile
            // (a rank whose wait ran out comes here too)
            __syncthreads();
            asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
            float *rows = reinterpret_cast<float *>(aA);  // [csize][ROWS]
            if (warp < 4) {
                uint32_t dst;
                asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(dst) : "r"(smem_u32(rows + crank * ROWS + tid)));
                asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst), "f"(v0 + v1 + spart[turn][tid]) : "memory");
            }
            asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
            if (crank == 0) {
                if (warp < 4) {
                    float sum = 0.f;
                    for (uint32_t k = 0; k < csize; ++k) sum += rows[k * ROWS + tid];
                    write_out(sum, t);
                }
                __syncthreads();  // before the activations are written again
            }
        }
        turn ^= 1;
        if (failed && csize == 1) break;
    }
    __syncthreads();
    if (warp < 4 && out_tile >= 0) write_out(out_sum + spart[turn ^ 1][tid], out_tile);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    if (__syncthreads_or(lost ? 1 : 0) && tid == 0) atomicOr(a.err, kErrTimeout);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(H));
}

template <bool LIST>
static cudaError_t launch(const Args &a, cudaStream_t st) {
    int dev = 0, sms = 0, sm_smem = 0;
    cudaFuncAttributes fa{};
    const int smem = smem_bytes(a.d, LIST);
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, masked_game_tc_kernel<LIST>);
    // the largest size this kernel can need, so that calls of different d on
    // different threads never lower each other's limit
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(masked_game_tc_kernel<LIST>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(32, LIST));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(masked_game_tc_kernel<LIST>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    // CTAs an SM holds, by registers (the launch bounds) and shared memory (1 KB
    // of it reserved per CTA); the occupancy query counts one for a kernel that
    // allocates tensor memory, of which these use a quarter each
    const int occ = std::min(LIST ? 2 : 3, sm_smem / (smem + (int)fa.sharedSizeBytes + 1024));
    // a persistent grid: the CTAs of an SM run their CUDA-core layers beside
    // each other's tensor-core waits
    const long long slots = (long long)std::max(1, occ) * sms;
    // background rows shared by the CTAs of a cluster where that shortens the
    // longest chain of passes (d = 12, 8 instances, 100 rows: 256 tiles)
    unsigned cluster = 1;
    auto chain = [&](long long c) {
        const long long groups = std::max<long long>(1, slots / c);
        return (a.n_tiles + groups - 1) / groups * ((a.n_bg + c - 1) / c);
    };
    for (unsigned c = 2; c <= MAX_CLUSTER && (int)c <= a.n_bg; ++c)
        if (chain(c) < chain(cluster)) cluster = c;
    const long long groups = std::min<long long>(a.n_tiles, std::max<long long>(1, slots / cluster));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(groups * cluster));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, masked_game_tc_kernel<LIST>, a);
}

}  // namespace ttfsi_mgtc

extern "C" tt_fsi_status tt_fsi_masked_game_tc_interventional(const tt_fsi_mlp *model, const double *x_dev,
                                                             const double *background_dev, int n_background,
                                                             int64_t B, const unsigned *coal_dev, int K,
                                                             float *out_dev, int *err_dev, struct CUstream_st *stream);

extern "C" tt_fsi_status tt_fsi_masked_game_tc(const tt_fsi_mlp *model, const double *x_dev,
                                              const double *baseline_dev, int64_t B, const unsigned *coal_dev,
                                              int K, float *out_dev, int *err_dev, struct CUstream_st *stream) {
    // a baseline is the interventional value function with one background row
    return tt_fsi_masked_game_tc_interventional(model, x_dev, baseline_dev, 1, B, coal_dev, K, out_dev, err_dev,
                                                stream);
}

extern "C" tt_fsi_status tt_fsi_masked_game_tc_interventional(const tt_fsi_mlp *model, const double *x_dev,
                                                             const double *background_dev, int n_background,
                                                             int64_t B, const unsigned *coal_dev, int K,
                                                             float *out_dev, int *err_dev, struct CUstream_st *stream) {
    using namespace ttfsi_mgtc;
    const double *baseline_dev = background_dev;
    if (!model || B < 0 || n_background < 1) return TT_FSI_ERR_INVALID_ARG;
    if (B == 0) return TT_FSI_OK;
    if (!x_dev || !baseline_dev || !out_dev || !err_dev) return TT_FSI_ERR_INVALID_ARG;
    if (!model->W1f || !model->b1f || !model->W2f || !model->b2f || !model->W3f) return TT_FSI_ERR_INVALID_ARG;
    if (model->h1 != H || model->h2 != H) return TT_FSI_ERR_UNSUPPORTED;
    if (coal_dev) {
        if (K < 1 || model->d < 1 || model->d > 32) return TT_FSI_ERR_INVALID_ARG;
    } else if (model->d < 7 || model->d > 30) {
        return TT_FSI_ERR_UNSUPPORTED;  // a dense tile is 128 coalitions of one instance
    }
    Args a{};
    a.W1 = model->W1f;
    a.b1 = model->b1f;
    a.W2 = model->W2f;
    a.b2 = model->b2f;
    a.W3 = model->W3f;
    a.b3 = (float)model->b3;
    a.x = x_dev;
    a.base = baseline_dev;
    a.n_bg = n_background;
    a.d = model->d;
    a.coal = coal_dev;
    a.K = coal_dev ? K : 0;
    a.out = out_dev;
    a.n_rows = coal_dev ? B * (long long)K : (B << model->d);
    a.n_tiles = (a.n_rows + ROWS - 1) / ROWS;
    a.err = err_dev;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    return (coal_dev ? launch<true>(a, st) : launch<false>(a, st)) == cudaSuccess ? TT_FSI_OK : TT_FSI_ERR_CUDA;
}
