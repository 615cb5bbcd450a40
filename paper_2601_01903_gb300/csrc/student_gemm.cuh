// The student's matrix products on the tcgen05 tensor cores, one or two
// independent products per launch, every operand read in the row-major layout
// its producer wrote:
//
//   C[M, N] = opA . opB,   A stored [M, K] (a_mn = 0) or [K, M] (a_mn = 1),
//                          B stored [N, K] (b_mn = 0) or [K, N] (b_mn = 1),
//
// BF16 operands, FP32 accumulators in tensor memory.  The tensor cores read a
// K-major or an MN-major tile equally well, so the backward products need no
// transposed copies of activations, gradients and weights (five 8 MB arrays
// written and read back per step at 4096 x 1024).
//
// One CTA of 8 warps computes a 128 x 128 tile of one K slice: one thread
// issues TMA loads into 32 KB stages, one issues the MMAs, all warps run
// the epilogue, each on 32 rows x 64 columns.  Two stages and 85 registers
// keep three CTAs on an SM, whose epilogues and main loops overlap; a launch
// with fewer CTAs takes more stages.
// The epilogue costs more than the products (a tile of layer 2 takes 4096
// clocks of tensor work and writes 96 KB): results go from registers through
// the idle stages, in the swizzled order of a TMA store, and leave as whole
// lines; the pre-activations of a GELU factor come in the same way.  Bias
// gradients are summed here too, from the FP32 values before they are rounded,
// so those values are never written out.
//
// One GB300, 4096 x 1024: layer 1 16.9 -> 9.3 us, layer 2 25.2 -> 14.5, dH2 23.7
// and dW3 17.7 -> 12.4 together, dH1 28.7, dW2 28.2 and dW1 14.4 -> 21.5 together
// (gemm_bf16_tcgen05_tma with its slice sums before).  No unit is saturated
// (tensor pipe 2 to 31 %, issue 13 to 36 %); alone, a launch has some 7 us of
// fixed costs (prologue, first load, drain), part of which the programmatic
// chain hides.
//
// Every wait on an mbarrier is bounded; a CTA whose wait runs out records
// kErrGemmTimeout, waits (bounded) for its loads in flight, frees its tensor
// memory and returns.
#pragma once

#include "gemm_tcgen05.cuh"

namespace ttfsi_sgemm {

using namespace ttfsi_gemm;

constexpr int SG_MAX_STAGES = 6;  // of 32 KB
constexpr int SG_THREADS = 256;
__host__ __device__ constexpr int sg_smem(int stages) { return stages * 2 * TILE_BYTES + 1024; }
// A CTA's loads are bound by their latency (two stages in flight: a tile of 16
// K blocks takes 14 us alone on its SM), so a launch takes as many stages as
// fit with the CTAs per SM that it has.
inline int sg_stages(int blocks, int sms) { return blocks <= sms ? 6 : blocks <= 2 * sms ? 3 : 2; }

enum : int { kPartial = 0, kAct = 1, kDgelu = 2 };

// One product.  kPartial: the raw FP32 tile of K slice z goes to rows
// z zrows .. of F.  kAct: z = acc + bias, F = z (when has_f), Hb = BF16
// GELU(z).  kDgelu: g = acc gelu'(Z), Hb = BF16 g, and the column sums of g
// over the tile's rows go to colpart[m tile][N].  With dwx, kDgelu multiplies
// the tile, as it lies in shared memory, by its rows of X (a second product on
// the tensor cores) and writes dwpart[m tile][N][xd], the tile's part of the
// weight gradient below; g itself then stays on the chip.
struct Job {
    CUtensorMap A, B;  // boxes of 64 x 128 (K-major) or 64 x 64 (MN-major) elements
    CUtensorMap F;     // FP32 output, boxes of 32 x 32
    CUtensorMap Hb;    // BF16 output, boxes of 64 x 32
    CUtensorMap Z;     // FP32 pre-activations, boxes of 32 x 32
    CUtensorMap X;     // BF16 instances [M, xd], boxes of 64 x 128
    const float *bias;
    float *colpart;
    int M, N, K;
    int a_mn, b_mn;
    int kind, has_f;
    int dwx, xd;  // xd: a multiple of 8, at most 64
    float *dwpart;
    int kbc;     // K blocks of 64 per slice
    int zrows;   // rows between slices of F, a multiple of 32 no less than M rounded up to 32
    int tiles_n, tiles_m;
    int blocks;  // tiles_n * tiles_m * slices
};
struct Jobs {
    Job j[2];
    int *err;
    int stages;  // sg_stages
};

__device__ __forceinline__ void tma_store_2d(const void *tmap, uint32_t src, int x, int y) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(tmap), "r"(x),
                 "r"(y), "r"(src)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap *m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory");
}

__device__ __forceinline__ void st_shared4(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}

__device__ __forceinline__ float4 ld_shared4(uint32_t a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(a)
                 : "memory");
    return v;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&p);
}

// ---- GELU and its derivative of packed FP32 pairs: the formula of
// normal_cdf_pdf, half its instructions ----
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f2 v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
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
__device__ __forceinline__ f2 both(float c) { return pack2(c, c); }

// q = erfc(|z| / sqrt 2) / 2 and e = exp(-z^2 / 2)
__device__ __forceinline__ void normal_tail2(f2 z, f2 &q, f2 &e) {
    const f2 x = mul2(z & 0x7fffffff7fffffffull, both(0.70710678118654752f));
    float a, b;
    unpack2(fma2(both(0.3275911f), x, both(1.0f)), a, b);
    asm("rcp.approx.ftz.f32 %0, %0;" : "+f"(a));
    asm("rcp.approx.ftz.f32 %0, %0;" : "+f"(b));
    const f2 t = pack2(a, b);
    f2 p = fma2(both(0.5f * 1.061405429f), t, both(0.5f * -1.453152027f));
    p = fma2(p, t, both(0.5f * 1.421413741f));
    p = fma2(p, t, both(0.5f * -0.284496736f));
    p = fma2(p, t, both(0.5f * 0.254829592f));
    unpack2(mul2(mul2(x, x), both(-1.4426950408889634f)), a, b);
    asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(a));
    asm("ex2.approx.ftz.f32 %0, %0;" : "+f"(b));
    e = pack2(a, b);
    q = mul2(mul2(p, t), e);
}

__device__ __forceinline__ f2 normal_cdf2(float z0, float z1, f2 q) {
    float q0, q1;
    unpack2(q, q0, q1);
    return pack2(z0 >= 0.f ? 1.0f - q0 : q0, z1 >= 0.f ? 1.0f - q1 : q1);
}

// z Phi(z), rounded to BF16
__device__ __forceinline__ uint32_t gelu_pair(float z0, float z1) {
    const f2 z = pack2(z0, z1);
    f2 q, e;
    normal_tail2(z, q, e);
    float y0, y1;
    unpack2(mul2(z, normal_cdf2(z0, z1, q)), y0, y1);
    return pack_bf16(y0, y1);
}

// v0, v1 times d/dz [z Phi(z)] = Phi(z) + z phi(z)
__device__ __forceinline__ void scale_gelu_grad(float &v0, float &v1, float z0, float z1) {
    const f2 z = pack2(z0, z1);
    f2 q, e;
    normal_tail2(z, q, e);
    const f2 pdf = mul2(both(0.39894228040143268f), e);
    unpack2(mul2(pack2(v0, v1), fma2(z, pdf, normal_cdf2(z0, z1, q))), v0, v1);
}

// 32 accumulator columns of the lane's row.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Shared-memory descriptor of an MN-major operand, 128-byte swizzle: 64
// elements of M or N by 8 of K per 1024-byte group; the next 8 of K follow
// (stride byte offset), the next 64 of M or N start `next` bytes on (leading
// byte offset; one 64 x 64 box each).
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t addr, uint32_t next = 8192) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)(next >> 4) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__global__ void __launch_bounds__(SG_THREADS, 3) student_gemm_kernel(const __grid_constant__ Jobs jobs) {
    extern __shared__ __align__(1024) unsigned char sg_raw[];
    const uint32_t base = (smem_u32(sg_raw) + 1023) & ~1023u;
    __shared__ __align__(8) uint64_t full[SG_MAX_STAGES], empty[SG_MAX_STAGES], done, zbar[8], xbar, xdone;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int s_fail;
    __shared__ float red[4][BN];

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int which = (int)blockIdx.x >= jobs.j[0].blocks;
    const Job &a = jobs.j[which];
    int t = (int)blockIdx.x - (which ? jobs.j[0].blocks : 0);
    const int n0 = (t % a.tiles_n) * BN;
    t /= a.tiles_n;
    const int m0 = (t % a.tiles_m) * BM;
    const int slice = t / a.tiles_m;
    const int kb0 = slice * a.kbc;
    const int nk = min(a.kbc, (a.K + BK - 1) / BK - kb0);
    const int n_cols = min(BN, a.N - n0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < jobs.stages; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        mbar_init(smem_u32(&done), 1);
        for (int w = 0; w < 8; ++w) mbar_init(smem_u32(&zbar[w]), 1);
        mbar_init(smem_u32(&xbar), 1);
        mbar_init(smem_u32(&xdone), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_fail = 0;
    }
    if (threadIdx.x == 64) {  // the descriptors, ahead of their first use
        prefetch_map(&a.A);
        prefetch_map(&a.B);
        if (a.kind == kDgelu) prefetch_map(&a.Z);
        prefetch_map(a.kind == kPartial ? &a.F : a.dwx ? &a.X : &a.Hb);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_sh)),
                     "r"(BN));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_sh;
    // the next kernel may set itself up from here on; it waits for this one to complete before it reads
    pdl_launch();
    pdl_wait();

    auto tileA = [&](int s) { return base + (uint32_t)(s * 2) * TILE_BYTES; };
    auto tileB = [&](int s) { return base + (uint32_t)(s * 2 + 1) * TILE_BYTES; };

    // Warps 0 and 1 go through their loops whole and elect one lane for each
    // copy or MMA: the operands stay in uniform registers, where a branch on
    // the lane makes the compiler move them there under divergence (a K block
    // took 900 clocks of issue, 256 of tensor work).
    if (warp == 0) {
        // producer; an operand tile is two halves of 64 rows (or columns), 8 KB each,
        // the second half of B only where columns use it
        const bool b_one = a.b_mn && n_cols <= 64;
        const uint32_t bytes = (b_one ? TILE_BYTES / 2 : TILE_BYTES) + TILE_BYTES;
        const bool leader = elect_one();
        const int a_mn = a.a_mn, b_mn = a.b_mn, stages = jobs.stages;
        int kb = 0, s = 0;
        uint32_t use = 0;
        for (; kb < nk; ++kb) {
            if (use > 0 && !mbar_wait(smem_u32(&empty[s]), (use - 1) & 1u)) {
                if (leader) atomicOr(&s_fail, 1);
                break;
            }
            if (leader) {
                const uint32_t bar = smem_u32(&full[s]);
                mbar_expect_tx(bar, bytes);
                const int k0 = (kb0 + kb) * BK;
                const uint32_t ta = tileA(s), tb = tileB(s);
                if (a_mn) {
                    tma_load_2d(ta, &a.A, m0, k0, bar);
                    tma_load_2d(ta + TILE_BYTES / 2, &a.A, m0 + 64, k0, bar);
                } else {
                    tma_load_2d(ta, &a.A, k0, m0, bar);
                }
                if (b_mn) {
                    tma_load_2d(tb, &a.B, n0, k0, bar);
                    if (!b_one) tma_load_2d(tb + TILE_BYTES / 2, &a.B, n0 + 64, k0, bar);
                } else {
                    tma_load_2d(tb, &a.B, k0, n0, bar);
                }
            }
            __syncwarp();
            if (++s == stages) {
                s = 0;
                ++use;
            }
        }
        if (kb < nk)  // gave up: let the loads in flight land before the CTA ends
            for (int i = max(0, kb - stages); i < kb; ++i)
                mbar_wait(smem_u32(&full[i % stages]), (uint32_t)(i / stages) & 1u);
        __syncwarp();
    } else if (warp == 1) {
        // MMA issuer: as many columns as the tile has, in sixteens (K beyond the
        // operands was filled with zeros)
        const uint32_t idesc =
            instr_desc_bf16(BM, (n_cols + 15) & ~15) | ((uint32_t)a.a_mn << 15) | ((uint32_t)a.b_mn << 16);
        const uint32_t stepA = (a.a_mn ? 2048u : 32u) >> 4, stepB = (a.b_mn ? 2048u : 32u) >> 4;
        const uint64_t da0 = a.a_mn ? smem_desc_mn(tileA(0)) : smem_desc(tileA(0));
        const uint64_t db0 = a.b_mn ? smem_desc_mn(tileB(0)) : smem_desc(tileB(0));
        const int stages = jobs.stages;
        const bool leader = elect_one();
        bool ok = true;
        int s = 0;
        uint32_t parity = 0;
        for (int kb = 0; kb < nk; ++kb) {
            if (!mbar_wait(smem_u32(&full[s]), parity)) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (leader) {
                const uint64_t da = da0 + (uint32_t)(s * (2 * TILE_BYTES >> 4));
                const uint64_t db = db0 + (uint32_t)(s * (2 * TILE_BYTES >> 4));
#pragma unroll
                for (int k16 = 0; k16 < BK / 16; ++k16)
                    mma_bf16(tmem, da + k16 * stepA, db + k16 * stepB, idesc, (kb > 0 || k16 > 0) ? 1u : 0u);
                mma_commit(smem_u32(&empty[s]));
            }
            __syncwarp();
            if (++s == stages) {
                s = 0;
                parity ^= 1u;
            }
        }
        if (leader) {
            if (!ok) atomicOr(&s_fail, 1);
            mma_commit(smem_u32(&done));  // arrives once every MMA issued above has completed
        }
        __syncwarp();
    }
    if (lane == 0 && !mbar_wait(smem_u32(&done), 0)) atomicOr(&s_fail, 1);
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    // Epilogue.  Warp w: rows 32 (w & 3) .., columns 64 (w >> 2) .., through
    // its own 8 KB of the idle stages (two 32 x 128-byte blocks, 32 KB apart; row
    // r's 16-byte chunk c at chunk c ^ (r & 7), the order of a 128-byte-swizzled
    // TMA copy).  A lane touches its own row only, so no lane waits for another.
    constexpr uint32_t kNext = 32768;
    const int q = warp & 3, row0 = m0 + 32 * q, colw = 64 * (warp >> 2);
    const uint32_t buf = base + (uint32_t)warp * 4096;
    const uint32_t line = buf + (uint32_t)lane * 128;
    const uint32_t sw = (uint32_t)(lane & 7);
    const bool fail = s_fail != 0;
    const int kind = a.kind;
    if (!fail && row0 < a.M && colw < n_cols) {
        const int nj = colw + 32 < n_cols ? 2 : 1;
        const uint32_t trow = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)colw;
        const int col0 = n0 + colw;
        if (kind == kPartial) {
            for (int j = 0; j < nj; ++j) {
                float v[32];
                tmem_ld32(trow + 32 * j, v);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    st_shared4(line + j * kNext + ((c ^ sw) << 4), __float_as_uint(v[4 * c]), __float_as_uint(v[4 * c + 1]),
                               __float_as_uint(v[4 * c + 2]), __float_as_uint(v[4 * c + 3]));
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) tma_store_2d(&a.F, buf + j * kNext, col0 + 32 * j, slice * a.zrows + row0);
            }
        } else if (kind == kAct) {
            uint32_t y[32];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                if (j < nj) {
                    float v[32];
                    tmem_ld32(trow + 32 * j, v);
                    // N and the bias's offset are multiples of 4
                    const float4 *bias = reinterpret_cast<const float4 *>(a.bias + col0 + 32 * j);
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const float4 b = col0 + 32 * j + 4 * c < a.N ? bias[c] : make_float4(0.f, 0.f, 0.f, 0.f);
                        v[4 * c] += b.x;
                        v[4 * c + 1] += b.y;
                        v[4 * c + 2] += b.z;
                        v[4 * c + 3] += b.w;
                    }
                    if (a.has_f) {
#pragma unroll
                        for (int c = 0; c < 8; ++c)
                            st_shared4(line + j * kNext + ((c ^ sw) << 4), __float_as_uint(v[4 * c]),
                                       __float_as_uint(v[4 * c + 1]), __float_as_uint(v[4 * c + 2]),
                                       __float_as_uint(v[4 * c + 3]));
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) tma_store_2d(&a.F, buf + j * kNext, col0 + 32 * j, row0);
                    }
#pragma unroll
                    for (int i = 0; i < 16; ++i) y[16 * j + i] = gelu_pair(v[2 * i], v[2 * i + 1]);
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i) y[16 * j + i] = 0u;
                }
            }
            // the first block is free once its store has been read out
            if (lane == 0 && a.has_f) {
                if (nj == 2)
                    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                else
                    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            }
            __syncwarp();
#pragma unroll
            for (int c = 0; c < 8; ++c)
                st_shared4(line + ((c ^ sw) << 4), y[4 * c], y[4 * c + 1], y[4 * c + 2], y[4 * c + 3]);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) tma_store_2d(&a.Hb, buf, col0, row0);
        } else {
            const uint32_t bar = smem_u32(&zbar[warp]);
            if (lane == 0) {
                mbar_expect_tx(bar, 4096u * (uint32_t)nj);
                for (int j = 0; j < nj; ++j) tma_load_2d(buf + j * kNext, &a.Z, col0 + 32 * j, row0, bar);
            }
            __syncwarp();
            const bool ok = mbar_wait(bar, 0);
            if (!ok && lane == 0) atomicOr(jobs.err, kErrGemmTimeout);
            for (int j = 0; j < nj; ++j) {
                float v[32];
                tmem_ld32(trow + 32 * j, v);
                // row by row in place: the 64 bytes of BF16 results of half j
                // replace chunks 4 j .. of the first block, which half 0 has read
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float4 z = ld_shared4(line + j * kNext + ((c ^ sw) << 4));
                    scale_gelu_grad(v[4 * c], v[4 * c + 1], z.x, z.y);
                    scale_gelu_grad(v[4 * c + 2], v[4 * c + 3], z.z, z.w);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    st_shared4(line + (((4 * j + c) ^ sw) << 4), pack_bf16(v[8 * c], v[8 * c + 1]),
                               pack_bf16(v[8 * c + 2], v[8 * c + 3]), pack_bf16(v[8 * c + 4], v[8 * c + 5]),
                               pack_bf16(v[8 * c + 6], v[8 * c + 7]));
                // column sums over the warp's 32 rows: halve the columns a
                // lane keeps at each step, lane l ends with column l
#pragma unroll
                for (int o = 16; o >= 1; o >>= 1)
#pragma unroll
                    for (int i = 0; i < o; ++i) {
                        const bool up = lane & o;
                        const float send = up ? v[i] : v[i + o];
                        v[i] = (up ? v[i + o] : v[i]) + __shfl_xor_sync(0xffffffffu, send, o);
                    }
                red[q][colw + 32 * j + lane] = v[0];
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0 && ok && !a.dwx) tma_store_2d(&a.Hb, buf, col0, row0);
        }
    }
    if (!fail && kind == kDgelu) {
        if (row0 >= a.M) {
            red[q][colw + lane] = 0.0f;
            red[q][colw + 32 + lane] = 0.0f;
            if (a.dwx) {
#pragma unroll
                for (int c = 0; c < 8; ++c) st_shared4(line + (c << 4), 0u, 0u, 0u, 0u);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (a.dwx && threadIdx.x == 0) {
            // g^T X: the first blocks are the tile [128 rows][2 x 64 columns],
            // MN-major; X replaces the second ones, all read by now
            const uint32_t xs = base + kNext;
            mbar_expect_tx(smem_u32(&xbar), TILE_BYTES);
            tma_load_2d(xs, &a.X, 0, m0, smem_u32(&xbar));
            const bool ok = mbar_wait(smem_u32(&xbar), 0);
            if (!ok) atomicOr(jobs.err, kErrGemmTimeout);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t idesc = instr_desc_bf16(BM, (a.xd + 15) & ~15) | (1u << 15) | (1u << 16);
            if (ok)
                for (int k16 = 0; k16 < BM / 16; ++k16)
                    mma_bf16(tmem, smem_desc_mn(base + k16 * 2048, 16384), smem_desc_mn(xs + k16 * 2048), idesc,
                             k16 > 0 ? 1u : 0u);
            mma_commit(smem_u32(&xdone));
        }
        if ((int)threadIdx.x < n_cols)
            a.colpart[(long long)(m0 / BM) * a.N + n0 + threadIdx.x] =
                (red[0][threadIdx.x] + red[1][threadIdx.x]) + (red[2][threadIdx.x] + red[3][threadIdx.x]);
        __syncwarp();
        if (a.dwx && warp < 4) {
            if (!mbar_wait(smem_u32(&xdone), 0) && lane == 0) atomicOr(jobs.err, kErrGemmTimeout);
            __syncwarp();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int h = n0 + 32 * warp + lane;
            float *out = a.dwpart + ((long long)(m0 / BM) * a.N + h) * a.xd;
            for (int c0 = 0; c0 < a.xd; c0 += 32) {
                float v[32];
                tmem_ld32(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)c0, v);
                if (h < a.N)
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        if (c0 + 4 * c < a.xd)
                            *reinterpret_cast<float4 *>(out + c0 + 4 * c) =
                                make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
            }
        }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (s_fail && threadIdx.x == 0) atomicOr(jobs.err, kErrGemmTimeout);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(BN));
}

}  // namespace ttfsi_sgemm
