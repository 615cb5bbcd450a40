// Amortised FSI explainer ("student"): a GELU MLP that maps an instance x to
// its FSI scores, trained on (x, exact FSI of v_x) pairs, its products on the
// tensor cores (student_gemm.cuh).  A training step is eight launches: the
// instances to BF16, three layers forward, the projection with loss and output
// gradient, [dH2 | dW3], [dW2 | dH1 with dW1], and the sums of partial results
// with Adam.  One GB300, 4096 instances, 1024 hidden units, 137 scores: 79 us
// (0.236 ms with 20 launches, transposed copies and separate sums).  This file
// also holds the launcher of the general BF16 GEMM (gemm_tcgen05.cuh) and its
// C ABI entry point.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>

#include "gemm_tcgen05.cuh"
#include "student_gemm.cuh"
#include "tt_fsi.h"

namespace {

tt_fsi_status st_status(cudaError_t e) {
    if (e == cudaSuccess) return TT_FSI_OK;
    return e == cudaErrorMemoryAllocation ? TT_FSI_ERR_NO_MEMORY : TT_FSI_ERR_CUDA;
}

std::atomic<bool> g_gemm_attr_set[64];

// The driver's tensor-map encoder, looked up through the runtime (so the
// library does not link the driver library itself); null if unavailable.
// Safe on several threads at once: each that finds none yet looks it up.
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static std::atomic<PFN_cuTensorMapEncodeTiled_v12000> found{nullptr};
    PFN_cuTensorMapEncodeTiled_v12000 fn = found.load();
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        if (fn) found.store(fn);
    }
    return fn;
}

// Tensor map of a row-major array [rows, cols] with row pitch ld elements:
// 128-byte swizzle, zero fill outside.  The encoder wants a current context,
// which a thread has only after its first runtime call of some kinds: setting
// the device it has makes one current.
bool encode_map(CUtensorMap *map, CUtensorMapDataType type, int elem, const void *ptr, long long rows, int cols, int ld,
                int box_cols, int box_rows, CUtensorMapL2promotion promotion = CU_TENSOR_MAP_L2_PROMOTION_L2_256B) {
    PFN_cuTensorMapEncodeTiled_v12000 encode = tensor_map_encoder();
    if (!encode) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * elem};
    const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    auto made = [&] {
        return encode(map, type, 2, const_cast<void *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                      CU_TENSOR_MAP_SWIZZLE_128B, promotion, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    int dev = 0;
    return made() || (cudaGetDevice(&dev) == cudaSuccess && cudaSetDevice(dev) == cudaSuccess && made());
}

// A BF16 operand [rows, K] of the GEMM: boxes of 128 x 64.
bool operand_tensor_map(CUtensorMap *map, const __nv_bfloat16 *ptr, int rows, int K, int ld) {
    return encode_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ptr, rows, K, ld, ttfsi_gemm::BK, ttfsi_gemm::BM,
                      CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
}

// Launches the TMA-fed kernel, or the cp.async kernel where an operand has
// no valid tensor map (the two compute the same products).
tt_fsi_status gemm_launch(const ttfsi_gemm::GemmArgs &a, cudaStream_t st) {
    using namespace ttfsi_gemm;
    if (a.M <= 0 || a.N <= 0 || a.K <= 0) return TT_FSI_OK;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return TT_FSI_ERR_CUDA;
    if (dev >= 0 && dev < 64 && !g_gemm_attr_set[dev]) {
        cudaError_t e = cudaFuncSetAttribute(gemm_bf16_tcgen05, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(gemm_bf16_tcgen05_tma, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     TMA_SMEM_BYTES);
        if (e != cudaSuccess) return st_status(e);
        g_gemm_attr_set[dev] = true;
    }
    dim3 grid((unsigned)((a.N + BN - 1) / BN), (unsigned)((a.M + BM - 1) / BM));
    CUtensorMap tmA, tmB;
    if (operand_tensor_map(&tmA, a.A, a.M, a.K, a.lda) && operand_tensor_map(&tmB, a.B, a.N, a.K, a.ldb))
        gemm_bf16_tcgen05_tma<<<grid, TMA_THREADS, TMA_SMEM_BYTES, st>>>(a, tmA, tmB);
    else
        gemm_bf16_tcgen05<<<grid, THREADS, SMEM_BYTES, st>>>(a);
    return st_status(cudaGetLastError());
}

}  // namespace

extern "C" tt_fsi_status tt_fsi_gemm_bf16(const void *A, int lda, const void *B, int ldb, int M, int N, int K,
                                          const float *bias, int act, const float *dgelu_z, int ldz, float *Cf,
                                          int ldcf, void *Cb, int ldcb, void *Ct, int ldct, int *err_dev,
                                          struct CUstream_st *stream) {
    if (M < 0 || N < 0 || K < 0 || !A || !B || !err_dev) return TT_FSI_ERR_INVALID_ARG;
    if ((lda % 8) || (ldb % 8) || lda < K || ldb < K) return TT_FSI_ERR_INVALID_ARG;  // 16-byte rows
    if ((((uintptr_t)A) | ((uintptr_t)B)) & 15) return TT_FSI_ERR_INVALID_ARG;
    if (act != 0 && act != 1) return TT_FSI_ERR_INVALID_ARG;
    ttfsi_gemm::GemmArgs a{};
    a.A = static_cast<const __nv_bfloat16 *>(A);
    a.B = static_cast<const __nv_bfloat16 *>(B);
    a.lda = lda;
    a.ldb = ldb;
    a.M = M;
    a.N = N;
    a.K = K;
    a.bias = bias;
    a.act = act;
    a.dgelu_z = dgelu_z;
    a.ldz = ldz;
    a.Cf = Cf;
    a.ldcf = ldcf;
    a.Cb = static_cast<__nv_bfloat16 *>(Cb);
    a.ldcb = ldcb;
    a.Ct = static_cast<__nv_bfloat16 *>(Ct);
    a.ldct = ldct;
    a.err = err_dev;
    return gemm_launch(a, reinterpret_cast<cudaStream_t>(stream));
}

// ============================================================================
// Student network d -> H -> H -> n_out (GELU), BF16 operands on the tensor
// cores, FP32 master weights and Adam state, output projected onto the
// efficiency constraint.
// ============================================================================
#include <cmath>
#include <cstring>
#include <new>
#include <utility>
#include <vector>

namespace ttfsi_student {

using bf16 = __nv_bfloat16;

// BF16 copies of up to three FP32 arrays (the weights on load, a batch of
// instances), one launch: element i of the concatenation.
struct CastJobs {
    const float *src[3];
    bf16 *dst[3];
    long long n[3];
};
__global__ void to_bf16_kernel(CastJobs c) {
    ttfsi_sgemm::pdl_launch();
    ttfsi_sgemm::pdl_wait();
    const long long step = (long long)gridDim.x * blockDim.x;
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    for (int k = 0; k < 3; ++k) {
        for (; i < c.n[k]; i += step) c.dst[k][i] = __float2bfloat16_rn(c.src[k][i]);
        i -= c.n[k];
    }
}

// Output layer and projection onto sum_{S != empty} phi(S) = target,
// phi(empty) = v_empty: y = the K slices of A2 W3^T added in order, plus b3.
// With labels also the squared-error loss and its gradient with respect to the
// raw outputs, dL/dY = P (2 (phi_p - phi) / (B n_out)), P = I - 11^T/(n_out-1)
// on the non-empty coordinates, 0 on the empty one, as BF16 (the operand of
// the backward products), its FP32 column sums over the block's rows (the bias
// gradient's partial sums) and the block's loss.  A warp takes a row, a block
// 8; the first 256 columns of y and the labels stay in registers over the three
// passes, the rest of y in the first slice's row, which only its own lanes
// read (a step of 4096 x 137 81.3 us with all of them re-read, 79.0 us so; bound by
// the latency of its loads, 27 warps per SM in one wave).
struct ProjectArgs {
    float *Y;  // [slices][zrows][ldy]
    int slices, ldy;
    long long zstride;
    const float *bias;
    int B, n_out;
    const float *target;
    float v_empty;
    float *phi;           // [B, n_out], or null
    const float *labels;  // [B, n_out], or null: no loss, no gradient
    float *loss_part, *col_part;  // [blocks], [blocks][n_out]
    bf16 *dYb;
    int ld_dyb;
};

__device__ __forceinline__ float warp_sum(float s) {
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

__global__ void __launch_bounds__(256) project_kernel(const ProjectArgs a) {
    constexpr int C = 4, CW = 32 * C;  // columns per lane and per warp in flight
    constexpr int KEEP = 2;            // chunks of CW columns held in registers
    __shared__ float red[8][CW];
    __shared__ float lred[8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = blockIdx.x * 8 + warp, n_out = a.n_out;
    const bool in = row < a.B;
    ttfsi_sgemm::pdl_launch();
    ttfsi_sgemm::pdl_wait();
    float *Y = a.Y + (long long)(in ? row : 0) * a.ldy;
    const long long at = (long long)(in ? row : 0) * n_out;
    // columns k0 + 32 c of the row: raw outputs (the slices' sum plus the bias), labels
    auto outputs = [&](int k0, float (&y)[C]) {
#pragma unroll
        for (int c = 0; c < C; ++c) y[c] = 0.f;
#pragma unroll 4
        for (int z = 0; z < a.slices; ++z)
#pragma unroll
            for (int c = 0; c < C; ++c) y[c] += Y[z * a.zstride + min(k0 + 32 * c, n_out - 1)];
#pragma unroll
        for (int c = 0; c < C; ++c) y[c] += a.bias[min(k0 + 32 * c, n_out - 1)];
    };
    auto labels = [&](int k0, float (&l)[C]) {
#pragma unroll
        for (int c = 0; c < C; ++c) l[c] = a.labels ? a.labels[at + min(k0 + 32 * c, n_out - 1)] : 0.f;
    };
    auto kept_outputs = [&](int k0, float (&y)[C]) {
#pragma unroll
        for (int c = 0; c < C; ++c) y[c] = Y[min(k0 + 32 * c, n_out - 1)];
    };

    float yk[KEEP][C] = {}, lk[KEEP][C] = {};
    float sum = 0.f;
    auto add_outputs = [&](int k0, const float (&y)[C]) {
#pragma unroll
        for (int c = 0; c < C; ++c)
            if (k0 + 32 * c > 0 && k0 + 32 * c < n_out) sum += y[c];
    };
    if (in) {
#pragma unroll
        for (int h = 0; h < KEEP; ++h)
            if (h * CW < n_out) {
                outputs(h * CW + lane, yk[h]);
                labels(h * CW + lane, lk[h]);
            }
#pragma unroll
        for (int h = 0; h < KEEP; ++h) add_outputs(h * CW + lane, yk[h]);
        for (int k0 = KEEP * CW + lane; k0 < n_out; k0 += CW) {
            float y[C];
            outputs(k0, y);
            add_outputs(k0, y);
#pragma unroll
            for (int c = 0; c < C; ++c)
                if (k0 + 32 * c < n_out) Y[k0 + 32 * c] = y[c];
        }
    }
    const float shift = in ? (a.target[row] - warp_sum(sum)) / (float)(n_out - 1) : 0.f;
    const float scale = 2.0f / ((float)a.B * (float)n_out);
    float loss = 0.f, gsum = 0.f;
    auto project = [&](int k0, const float (&y)[C], const float (&l)[C]) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = k0 + 32 * c;
            if (k >= n_out) break;
            const float p = (k == 0) ? a.v_empty : y[c] + shift;
            if (a.phi) a.phi[at + k] = p;
            const float e = p - l[c];
            loss += e * e;
            if (k > 0) gsum += scale * e;
        }
    };
    if (in) {
#pragma unroll
        for (int h = 0; h < KEEP; ++h) project(h * CW + lane, yk[h], lk[h]);
        for (int k0 = KEEP * CW + lane; k0 < n_out; k0 += CW) {
            float y[C], l[C];
            kept_outputs(k0, y);
            labels(k0, l);
            project(k0, y, l);
        }
    }
    if (!a.labels) return;
    const float gmean = warp_sum(gsum) / (float)(n_out - 1);
    loss = warp_sum(loss);
    if (lane == 0) lred[warp] = loss;
    auto gradient = [&](int k1, const float (&y)[C], const float (&l)[C]) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = k1 + 32 * c + lane;
            float g = 0.f;
            if (in && k > 0 && k < n_out) g = scale * (y[c] + shift - l[c]) - gmean;
            if (in && k < a.ld_dyb) a.dYb[(long long)row * a.ld_dyb + k] = __float2bfloat16_rn(g);
            red[warp][32 * c + lane] = g;
        }
        __syncthreads();
        const int k = k1 + (int)threadIdx.x;
        if ((int)threadIdx.x < CW && k < n_out) {
            float t = 0.f;
#pragma unroll
            for (int w = 0; w < 8; ++w) t += red[w][threadIdx.x];
            a.col_part[(long long)blockIdx.x * n_out + k] = t;
        }
        __syncthreads();
    };
#pragma unroll
    for (int h = 0; h < KEEP; ++h)
        if (h * CW < a.ld_dyb) gradient(h * CW, yk[h], lk[h]);
    for (int k1 = KEEP * CW; k1 < a.ld_dyb; k1 += CW) {
        float y[C], l[C];
        kept_outputs(k1 + lane, y);
        labels(k1 + lane, l);
        gradient(k1, y, l);
    }
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < 8; ++w) t += lred[w];
        a.loss_part[blockIdx.x] = t;
    }
}

// The end of a step: every gradient is the sum of partial results in a fixed
// order (K slices of the weight gradients, row blocks of the bias gradients),
// and with `update` Adam (Kingma & Ba) follows on the spot, m = b1 m +
// (1-b1) g, v = b2 v + (1-b2) g^2, p -= lr (m / (1 - b1^t)) / (sqrt(v /
// (1 - b2^t)) + eps), with the BF16 copy of a weight that the products read.
// Four weights per thread; a block per 32 columns of a bias, its warps over
// the row blocks; the first block adds the loss.
struct FinishArgs {
    float *p, *m, *v, *g;
    const float *wpart[3];  // [slices][stride]
    long long wstride[3];
    int wslices[3];
    long long woff[3], wn[3];  // multiples of 4
    bf16 *wb[3];
    const float *bpart[3];  // [parts][bn]
    int bparts[3], bn[3];
    long long boff[3];
    const float *loss_part;
    int loss_parts;
    float loss_scale;
    float *loss;  // or null
    int bias_blocks;  // the loss's and the biases' blocks, ahead of the weights'
    int update;
    float lr, b1, b2, eps, c1, c2;
};

__device__ __forceinline__ float adam_one(const FinishArgs &a, float g, float &m, float &v, float p) {
    m = a.b1 * m + (1.f - a.b1) * g;
    v = a.b2 * v + (1.f - a.b2) * g * g;
    return p - a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
}

__global__ void __launch_bounds__(256) finish_kernel(const __grid_constant__ FinishArgs a) {
    __shared__ float red[8][32];
    ttfsi_sgemm::pdl_launch();
    ttfsi_sgemm::pdl_wait();
    if ((int)blockIdx.x < a.bias_blocks) {
        const int lane = threadIdx.x & 31;
        const int warp = threadIdx.x >> 5;
        int w = (int)blockIdx.x - 1, k = 0;
        while (w >= 0 && k < 3 && w >= (a.bn[k] + 31) / 32) w -= (a.bn[k++] + 31) / 32;
        const int c = w * 32 + lane;
        float g = 0.f;
        if (w < 0) {  // the loss
            for (int i = threadIdx.x; i < a.loss_parts; i += 256) g += a.loss_part[i];
            g = warp_sum(g);
        } else if (c < a.bn[k]) {
#pragma unroll 8
            for (int i = warp; i < a.bparts[k]; i += 8) g += a.bpart[k][(long long)i * a.bn[k] + c];
        }
        red[warp][lane] = g;
        __syncthreads();
        if (warp > 0) return;
        g = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) g += red[i][lane];
        if (w < 0) {
            if (lane == 0 && a.loss) *a.loss = g * a.loss_scale;
            return;
        }
        if (c >= a.bn[k]) return;
        const long long at = a.boff[k] + c;
        a.g[at] = g;
        if (a.update) {
            float m = a.m[at], v = a.v[at];
            a.p[at] = adam_one(a, g, m, v, a.p[at]);
            a.m[at] = m;
            a.v[at] = v;
        }
        return;
    }
    long long i = ((long long)(blockIdx.x - a.bias_blocks) * 256 + threadIdx.x) * 4;
    int k = 0;
    while (k < 3 && i >= a.wn[k]) i -= a.wn[k++];
    if (k >= 3) return;
    const long long at = a.woff[k] + i;
    float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
    for (int z = 0; z < a.wslices[k]; ++z) {
        const float4 x = *reinterpret_cast<const float4 *>(a.wpart[k] + z * a.wstride[k] + i);
        g.x += x.x;
        g.y += x.y;
        g.z += x.z;
        g.w += x.w;
    }
    *reinterpret_cast<float4 *>(a.g + at) = g;
    if (!a.update) return;
    float4 m = *reinterpret_cast<float4 *>(a.m + at), v = *reinterpret_cast<float4 *>(a.v + at);
    float4 p = *reinterpret_cast<float4 *>(a.p + at);
    p.x = adam_one(a, g.x, m.x, v.x, p.x);
    p.y = adam_one(a, g.y, m.y, v.y, p.y);
    p.z = adam_one(a, g.z, m.z, v.z, p.z);
    p.w = adam_one(a, g.w, m.w, v.w, p.w);
    *reinterpret_cast<float4 *>(a.m + at) = m;
    *reinterpret_cast<float4 *>(a.v + at) = v;
    *reinterpret_cast<float4 *>(a.p + at) = p;
    uint2 b;
    b.x = ttfsi_sgemm::pack_bf16(p.x, p.y);
    b.y = ttfsi_sgemm::pack_bf16(p.z, p.w);
    *reinterpret_cast<uint2 *>(a.wb[k] + i) = b;
}

// Surrogate residual of each instance on its sampled coalitions:
// g(T) = sum over scores S subset of T of phi(S);
// r = sqrt(mean_k (g(T_k) - v(T_k))^2).  One warp per instance; a lane sums
// two coalitions at a time, so that a score and its mask, the same for all
// lanes, are read once for 64 of them, eight scores in flight (4096 instances,
// 64 coalitions, 137 scores: 15.9 us one coalition and one score at a time, 9.5
// us now).
__global__ void __launch_bounds__(256) residual_kernel(const float *phi, int B, int n_out, const unsigned *masks,
                                                       const unsigned *coal, const float *vcoal, int K, float *resid) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= B) return;
    const float *p = phi + (long long)warp * n_out;
    const unsigned *T = coal + (long long)warp * K;
    const float *v = vcoal + (long long)warp * K;
    float acc = 0.f;
    for (int k = lane; k < K; k += 64) {
        const bool two = k + 32 < K;
        const unsigned out0 = ~T[k], out1 = two ? ~T[k + 32] : 0u;
        const float v0 = v[k], v1 = two ? v[k + 32] : 0.f;
        float g0 = 0.f, g1 = 0.f;
        int q = 0;
        for (; q + 8 <= n_out; q += 8) {
            unsigned m[8];
            float f[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                m[i] = __ldg(masks + q + i);
                f[i] = __ldg(p + q + i);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (!(m[i] & out0)) g0 += f[i];
                if (!(m[i] & out1)) g1 += f[i];
            }
        }
        for (; q < n_out; ++q) {
            const unsigned m = __ldg(masks + q);
            const float f = __ldg(p + q);
            if (!(m & out0)) g0 += f;
            if (!(m & out1)) g1 += f;
        }
        const float e0 = g0 - v0;
        acc += e0 * e0;
        if (two) {
            const float e1 = g1 - v1;
            acc += e1 * e1;
        }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) resid[warp] = sqrtf(acc / (float)K);
}

int grid_for(long long n) {
    long long g = (n + 255) / 256;
    if (g > 4096) g = 4096;
    return (int)(g < 1 ? 1 : g);
}

}  // namespace ttfsi_student

struct tt_fsi_student_s {
    int d = 0, H = 0, n_out = 0, n_pad = 0, max_batch = 0, ldy = 0, sms = 152;
    long long n_params = 0;
    long long off_W1 = 0, off_b1 = 0, off_W2 = 0, off_b2 = 0, off_W3 = 0, off_b3 = 0;
    float *params = nullptr, *m = nullptr, *v = nullptr, *grads = nullptr;
    __nv_bfloat16 *W1b = nullptr, *W2b = nullptr, *W3b = nullptr;
    __nv_bfloat16 *Xb = nullptr, *A1 = nullptr, *A2 = nullptr, *dYb = nullptr, *dH2 = nullptr, *dH1 = nullptr;
    float *Z1 = nullptr, *Z2 = nullptr;
    float *Y = nullptr;                                            // K slices of the output layer
    float *part1 = nullptr, *part2 = nullptr, *part3 = nullptr;    // K slices of the weight gradients
    float *col1 = nullptr, *col2 = nullptr, *col3 = nullptr;       // row-block sums of the bias gradients
    float *loss_part = nullptr;
    int *err = nullptr;
    float lr = 1e-3f, beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
    long long step = 0;
    // the products of a batch of plan_B instances (their tensor maps name the
    // handle's own buffers and the batch's row count)
    int plan_B = 0;
    ttfsi_sgemm::Jobs f1_train, f1, f2_train, f2, f3, b3, b2, b1;
    std::vector<void *> allocs;
};

namespace {

using ttfsi_student::bf16;

template <typename T>
cudaError_t st_alloc(tt_fsi_student_s *s, T **p, size_t count) {
    cudaError_t e = cudaMalloc((void **)p, count * sizeof(T) + 16);
    if (e == cudaSuccess) {
        s->allocs.push_back(*p);
        e = cudaMemset(*p, 0, count * sizeof(T) + 16);
    }
    return e;
}

// Launches a kernel of the step as the programmatic dependent of the one
// before it: its CTAs are placed and set up while that one drains, and every
// kernel of the chain waits for the full completion of its predecessor
// (griddepcontrol.wait) before it reads or writes memory.
template <typename... P, typename... A>
tt_fsi_status chain(void (*kernel)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t st, A &&...args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return st_status(cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...));
}

// K slices of a product: enough for one tile per SM, at least 4 K blocks each.
// (A step of 4096 x 1024 with slices for 228 tiles, 152 and 128: 90.4, 81.3 and
// 80.8 us; 304 cost 13 us more than 152 did: the partial sums of more slices
// cost more than they overlap.)
void k_split(int sms, int M, int N, int K, int &kbc, int &slices) {
    using namespace ttfsi_gemm;
    const int tiles = ((M + BM - 1) / BM) * ((N + BN - 1) / BN), nk = (K + BK - 1) / BK;
    slices = std::max(1, std::min((sms + tiles - 1) / tiles, nk / 4));
    kbc = (nk + slices - 1) / slices;
    slices = (nk + kbc - 1) / kbc;
}

int round_up(int n, int to) { return (n + to - 1) / to * to; }

// A product of the step, in K slices for split_sms multiprocessors (0: one slice).
// op = 1: the operand is stored [K, rows].
bool make_job(ttfsi_sgemm::Job &j, const bf16 *A, int lda, int a_mn, const bf16 *B, int ldb, int b_mn, int M, int N,
              int K, int split_sms) {
    using namespace ttfsi_gemm;
    const auto T = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    j.M = M;
    j.N = N;
    j.K = K;
    j.a_mn = a_mn;
    j.b_mn = b_mn;
    j.tiles_m = (M + BM - 1) / BM;
    j.tiles_n = (N + BN - 1) / BN;
    int slices = 1;
    j.kbc = (K + BK - 1) / BK;
    if (split_sms) k_split(split_sms, M, N, K, j.kbc, slices);
    j.zrows = round_up(M, 32);
    j.blocks = j.tiles_m * j.tiles_n * slices;
    return (a_mn ? encode_map(&j.A, T, 2, A, K, M, lda, 64, BK) : encode_map(&j.A, T, 2, A, M, K, lda, BK, BM)) &&
           (b_mn ? encode_map(&j.B, T, 2, B, K, N, ldb, 64, BK) : encode_map(&j.B, T, 2, B, N, K, ldb, BK, BN));
}

int job_slices(const ttfsi_sgemm::Job &j) { return j.blocks / (j.tiles_m * j.tiles_n); }

bool out_partial(ttfsi_sgemm::Job &j, float *F, int ld) {
    j.kind = ttfsi_sgemm::kPartial;
    return encode_map(&j.F, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, F, (long long)j.zrows * job_slices(j), j.N, ld, 32, 32);
}

bool out_act(ttfsi_sgemm::Job &j, const float *bias, float *Z, bf16 *Hb) {
    j.kind = ttfsi_sgemm::kAct;
    j.bias = bias;
    j.has_f = Z != nullptr;
    return (!Z || encode_map(&j.F, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, Z, j.M, j.N, j.N, 32, 32)) &&
           encode_map(&j.Hb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Hb, j.M, j.N, j.N, 64, 32);
}

bool out_dgelu(ttfsi_sgemm::Job &j, const float *Z, bf16 *Hb, float *colpart) {
    j.kind = ttfsi_sgemm::kDgelu;
    j.colpart = colpart;
    return encode_map(&j.Z, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, Z, j.M, j.N, j.N, 32, 32) &&
           (!Hb || encode_map(&j.Hb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Hb, j.M, j.N, j.N, 64, 32));
}

// dH1's product also forms its tile's part of dW1 = dH1^T X where a row of X
// fits one box (otherwise dH1 is written out and dW1 has a launch of its own;
// 4096 x 1024, d = 16: 92.6 us a step with it, 97.2 us without).
bool dw1_fused(const tt_fsi_student_s *s) { return s->d <= 64; }

bool out_dw(ttfsi_sgemm::Job &j, const bf16 *X, int d, float *dwpart) {
    j.dwx = 1;
    j.xd = d;
    j.dwpart = dwpart;
    return encode_map(&j.X, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, X, j.M, d, d, 64, ttfsi_gemm::BM);
}

// The products for batches of B instances; made again when B changes.
tt_fsi_status plan_batch(tt_fsi_student_s *s, int B) {
    if (s->plan_B == B) return TT_FSI_OK;
    s->plan_B = 0;
    const int d = s->d, H = s->H, n_out = s->n_out, n_pad = s->n_pad;
    const float *P = s->params;
    bool ok = true;
    for (auto *j : {&s->f1_train, &s->f1, &s->f2_train, &s->f2, &s->f3, &s->b3, &s->b2, &s->b1}) {
        memset(j, 0, sizeof(*j));
        j->err = s->err;
    }
    for (auto *j : {&s->f1_train, &s->f1})
        ok = ok && make_job(j->j[0], s->Xb, d, 0, s->W1b, d, 0, B, H, d, 0) &&
             out_act(j->j[0], P + s->off_b1, j == &s->f1_train ? s->Z1 : nullptr, s->A1);
    for (auto *j : {&s->f2_train, &s->f2})
        ok = ok && make_job(j->j[0], s->A1, H, 0, s->W2b, H, 0, B, H, H, 0) &&
             out_act(j->j[0], P + s->off_b2, j == &s->f2_train ? s->Z2 : nullptr, s->A2);
    ok = ok && make_job(s->f3.j[0], s->A2, H, 0, s->W3b, H, 0, B, n_out, H, s->sms) &&
         out_partial(s->f3.j[0], s->Y, s->ldy);
    // dH2 = (dY W3) gelu'(Z2) and dW3 = dY^T A2
    ok = ok && make_job(s->b3.j[0], s->dYb, n_pad, 0, s->W3b, H, 1, B, H, n_out, 0) &&
         out_dgelu(s->b3.j[0], s->Z2, s->dH2, s->col2) &&
         make_job(s->b3.j[1], s->dYb, n_pad, 1, s->A2, H, 1, n_out, H, B, s->sms) &&
         out_partial(s->b3.j[1], s->part3, H);
    // dW2 = dH2^T A1 and dH1 = (dH2 W2) gelu'(Z1)
    ok = ok && make_job(s->b2.j[0], s->dH2, H, 1, s->A1, H, 1, H, H, B, s->sms) &&
         out_partial(s->b2.j[0], s->part2, H) &&
         make_job(s->b2.j[1], s->dH2, H, 0, s->W2b, H, 1, B, H, H, 0) &&
         out_dgelu(s->b2.j[1], s->Z1, s->dH1, s->col1);
    // dW1 = dH1^T X
    if (dw1_fused(s))
        ok = ok && out_dw(s->b2.j[1], s->Xb, d, s->part1);
    else
        ok = ok && make_job(s->b1.j[0], s->dH1, H, 1, s->Xb, d, 1, H, d, B, s->sms) && out_partial(s->b1.j[0], s->part1, d);
    if (!ok) return TT_FSI_ERR_CUDA;
    for (auto *j : {&s->f1_train, &s->f1, &s->f2_train, &s->f2, &s->f3, &s->b3, &s->b2, &s->b1})
        j->stages = ttfsi_sgemm::sg_stages(j->j[0].blocks + j->j[1].blocks, s->sms);
    s->plan_B = B;
    return TT_FSI_OK;
}

tt_fsi_status run_jobs(const ttfsi_sgemm::Jobs &j, cudaStream_t st) {
    return chain(ttfsi_sgemm::student_gemm_kernel, (unsigned)(j.j[0].blocks + j.j[1].blocks), ttfsi_sgemm::SG_THREADS,
                 (size_t)ttfsi_sgemm::sg_smem(j.stages), st, j);
}

// BF16 copies of the three weight matrices (a step keeps them up to date itself).
tt_fsi_status refresh_bf16(tt_fsi_student_s *s, cudaStream_t st) {
    ttfsi_student::CastJobs c{};
    const long long H = s->H;
    c.src[0] = s->params + s->off_W1;
    c.dst[0] = s->W1b;
    c.n[0] = H * s->d;
    c.src[1] = s->params + s->off_W2;
    c.dst[1] = s->W2b;
    c.n[1] = H * H;
    c.src[2] = s->params + s->off_W3;
    c.dst[2] = s->W3b;
    c.n[2] = H * s->n_out;
    return chain(ttfsi_student::to_bf16_kernel, (unsigned)ttfsi_student::grid_for(c.n[0] + c.n[1] + c.n[2]), 256, 0, st,
                 c);
}

// Forward pass up to the K slices of the raw outputs; `train` also keeps the
// FP32 pre-activations, which only the backward pass reads.
tt_fsi_status forward(tt_fsi_student_s *s, const float *x, int B, bool train, cudaStream_t st) {
    tt_fsi_status r = plan_batch(s, B);
    if (r != TT_FSI_OK) return r;
    ttfsi_student::CastJobs c{};
    c.src[0] = x;
    c.dst[0] = s->Xb;
    c.n[0] = (long long)B * s->d;
    r = chain(ttfsi_student::to_bf16_kernel, (unsigned)ttfsi_student::grid_for(c.n[0]), 256, 0, st, c);
    if (r == TT_FSI_OK) r = run_jobs(train ? s->f1_train : s->f1, st);
    if (r == TT_FSI_OK) r = run_jobs(train ? s->f2_train : s->f2, st);
    if (r == TT_FSI_OK) r = run_jobs(s->f3, st);
    return r;
}

constexpr int kProjectRows = 8;  // rows per block of the projection

ttfsi_student::ProjectArgs project_args(tt_fsi_student_s *s, const float *target, float v_empty, int B) {
    const ttfsi_sgemm::Job &j = s->f3.j[0];
    ttfsi_student::ProjectArgs a{};
    a.Y = s->Y;
    a.slices = job_slices(j);
    a.ldy = s->ldy;
    a.zstride = (long long)j.zrows * s->ldy;
    a.bias = s->params + s->off_b3;
    a.B = B;
    a.n_out = s->n_out;
    a.target = target;
    a.v_empty = v_empty;
    return a;
}

// Forward, backward and the gradients (with `update`, Adam too).
tt_fsi_status step(tt_fsi_student_s *s, const float *x, const float *labels, const float *target, float v_empty, int B,
                   float *loss_dev, bool update, cudaStream_t st) {
    tt_fsi_status r = forward(s, x, B, true, st);
    if (r != TT_FSI_OK) return r;
    const int pblocks = (B + kProjectRows - 1) / kProjectRows, mtiles = (B + ttfsi_gemm::BM - 1) / ttfsi_gemm::BM;
    ttfsi_student::ProjectArgs p = project_args(s, target, v_empty, B);
    p.labels = labels;
    p.loss_part = s->loss_part;
    p.col_part = s->col3;
    p.dYb = s->dYb;
    p.ld_dyb = s->n_pad;
    r = chain(ttfsi_student::project_kernel, (unsigned)pblocks, 256, 0, st, p);
    if (r == TT_FSI_OK) r = run_jobs(s->b3, st);
    if (r == TT_FSI_OK) r = run_jobs(s->b2, st);
    if (r == TT_FSI_OK && !dw1_fused(s)) r = run_jobs(s->b1, st);
    if (r != TT_FSI_OK) return r;

    ttfsi_student::FinishArgs f{};
    f.p = s->params;
    f.m = s->m;
    f.v = s->v;
    f.g = s->grads;
    const ttfsi_sgemm::Job *jobs[3] = {&s->b1.j[0], &s->b2.j[0], &s->b3.j[1]};
    float *parts[3] = {s->part1, s->part2, s->part3}, *cols[3] = {s->col1, s->col2, s->col3};
    const long long woff[3] = {s->off_W1, s->off_W2, s->off_W3}, boff[3] = {s->off_b1, s->off_b2, s->off_b3};
    bf16 *wb[3] = {s->W1b, s->W2b, s->W3b};
    long long weights = 0;
    f.bias_blocks = 1;  // the loss
    for (int k = 0; k < 3; ++k) {
        f.wpart[k] = parts[k];
        if (k == 0 && dw1_fused(s)) {
            f.wslices[k] = mtiles;
            f.wn[k] = f.wstride[k] = (long long)s->H * s->d;
        } else {
            f.wslices[k] = job_slices(*jobs[k]);
            f.wn[k] = (long long)jobs[k]->M * jobs[k]->N;
            f.wstride[k] = (long long)jobs[k]->zrows * jobs[k]->N;
        }
        f.woff[k] = woff[k];
        f.wb[k] = wb[k];
        f.bpart[k] = cols[k];
        f.bparts[k] = k == 2 ? pblocks : mtiles;
        f.bn[k] = k == 2 ? s->n_out : s->H;
        f.boff[k] = boff[k];
        weights += f.wn[k];
        f.bias_blocks += (f.bn[k] + 31) / 32;
    }
    f.loss_part = s->loss_part;
    f.loss_parts = pblocks;
    f.loss_scale = 1.0f / ((float)B * s->n_out);
    f.loss = loss_dev;
    f.update = update;
    if (update) {
        s->step += 1;
        f.lr = s->lr;
        f.b1 = s->beta1;
        f.b2 = s->beta2;
        f.eps = s->eps;
        f.c1 = 1.0f - (float)std::pow((double)s->beta1, (double)s->step);
        f.c2 = 1.0f - (float)std::pow((double)s->beta2, (double)s->step);
    }
    return chain(ttfsi_student::finish_kernel, (unsigned)(f.bias_blocks + (weights / 4 + 255) / 256), 256, 0, st, f);
}

void student_free(tt_fsi_student_s *s) {
    for (void *p : s->allocs) cudaFree(p);
    s->allocs.clear();
}

}  // namespace

extern "C" {

tt_fsi_status tt_fsi_student_create(int d, int hidden, int n_out, int max_batch, const float *params_host,
                                    tt_fsi_student *out) {
    if (!out || !params_host || d < 1 || hidden < 8 || n_out < 2 || max_batch < 1) return TT_FSI_ERR_INVALID_ARG;
    if ((d % 8) || (hidden % 8)) return TT_FSI_ERR_UNSUPPORTED;  // 16-byte rows of the BF16 operands
    *out = nullptr;
    tt_fsi_student_s *s = new (std::nothrow) tt_fsi_student_s();
    if (!s) return TT_FSI_ERR_NO_MEMORY;
    s->d = d;
    s->H = hidden;
    s->n_out = n_out;
    s->n_pad = (n_out + 15) / 16 * 16;
    s->max_batch = max_batch;
    s->ldy = round_up(n_out, 4);  // 16-byte rows
    long long o = 0;
    s->off_W1 = o;
    o += (long long)hidden * d;
    s->off_b1 = o;
    o += hidden;
    s->off_W2 = o;
    o += (long long)hidden * hidden;
    s->off_b2 = o;
    o += hidden;
    s->off_W3 = o;
    o += (long long)n_out * hidden;
    s->off_b3 = o;
    o += n_out;
    s->n_params = o;
    const size_t Bm = (size_t)max_batch, H = (size_t)hidden;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&s->sms, cudaDevAttrMultiProcessorCount, dev);
    auto A = [&](auto **p, size_t n) {
        if (e == cudaSuccess) e = st_alloc(s, p, n);
    };
    A(&s->params, (size_t)o);
    A(&s->m, (size_t)o);
    A(&s->v, (size_t)o);
    A(&s->grads, (size_t)o);
    A(&s->W1b, H * d);
    A(&s->W2b, H * H);
    A(&s->W3b, (size_t)s->n_pad * H);
    A(&s->Xb, Bm * d);
    A(&s->A1, Bm * H);
    A(&s->A2, Bm * H);
    A(&s->Z1, Bm * H);
    A(&s->Z2, Bm * H);
    A(&s->dYb, Bm * s->n_pad);
    A(&s->dH2, Bm * H);
    if (!dw1_fused(s)) A(&s->dH1, Bm * H);
    const size_t mtiles = (Bm + ttfsi_gemm::BM - 1) / ttfsi_gemm::BM, pblocks = (Bm + kProjectRows - 1) / kProjectRows;
    A(&s->col1, mtiles * H);
    A(&s->col2, mtiles * H);
    A(&s->col3, pblocks * n_out);
    A(&s->loss_part, pblocks);
    {
        // K slices, for the batch size up to max_batch that needs most rows: a
        // weight gradient has most slices at the largest batch, the output
        // layer may have more of them at a smaller one
        int kbc, slices;
        auto rows = [&](int M, int N, int K) {
            k_split(s->sms, M, N, K, kbc, slices);
            return (size_t)slices * round_up(M, 32);
        };
        size_t y = 0, w[3] = {0, 0, 0};
        const int shape[3][2] = {{hidden, d}, {hidden, hidden}, {n_out, hidden}};
        for (int b = max_batch; b > 0; b -= std::min(b, 64)) {
            y = std::max(y, rows(b, n_out, hidden));
            for (int k = 0; k < 3; ++k) w[k] = std::max(w[k], rows(shape[k][0], shape[k][1], b));
        }
        for (int b = 128; b <= max_batch; b += 128) {
            y = std::max(y, rows(b, n_out, hidden));
            for (int k = 0; k < 3; ++k) w[k] = std::max(w[k], rows(shape[k][0], shape[k][1], b));
        }
        A(&s->Y, y * s->ldy);
        A(&s->part1, dw1_fused(s) ? mtiles * H * d : w[0] * d);
        A(&s->part2, w[1] * H);
        A(&s->part3, w[2] * H);
    }
    A(&s->err, 1);
    if (e == cudaSuccess) e = cudaMemcpy(s->params, params_host, (size_t)o * sizeof(float), cudaMemcpyHostToDevice);
    tt_fsi_status r = st_status(e);
    if (r == TT_FSI_OK)
        r = st_status(cudaFuncSetAttribute(ttfsi_sgemm::student_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           ttfsi_sgemm::sg_smem(ttfsi_sgemm::SG_MAX_STAGES)));
    if (r == TT_FSI_OK) r = refresh_bf16(s, nullptr);
    if (r == TT_FSI_OK) r = st_status(cudaDeviceSynchronize());
    if (r != TT_FSI_OK) {
        student_free(s);
        delete s;
        return r;
    }
    *out = s;
    return TT_FSI_OK;
}

void tt_fsi_student_destroy(tt_fsi_student s) {
    if (!s) return;
    cudaDeviceSynchronize();
    student_free(s);
    delete s;
}

int64_t tt_fsi_student_num_params(tt_fsi_student s) { return s ? s->n_params : -1; }

tt_fsi_status tt_fsi_student_set_adam(tt_fsi_student s, float lr, float beta1, float beta2, float eps) {
    if (!s || !(lr >= 0.f) || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f) || !(eps > 0.f))
        return TT_FSI_ERR_INVALID_ARG;
    s->lr = lr;
    s->beta1 = beta1;
    s->beta2 = beta2;
    s->eps = eps;
    return TT_FSI_OK;
}

tt_fsi_status tt_fsi_student_gradients(tt_fsi_student s, const float *x_dev, const float *labels_dev,
                                       const float *target_dev, float v_empty, int B, float *loss_dev,
                                       struct CUstream_st *stream) {
    if (!s || !x_dev || !labels_dev || !target_dev || B < 1 || B > s->max_batch) return TT_FSI_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    return step(s, x_dev, labels_dev, target_dev, v_empty, B, loss_dev, false, st);
}

tt_fsi_status tt_fsi_student_train_step(tt_fsi_student s, const float *x_dev, const float *labels_dev,
                                        const float *target_dev, float v_empty, int B, float *loss_dev,
                                        struct CUstream_st *stream) {
    if (!s || !x_dev || !labels_dev || !target_dev || B < 1 || B > s->max_batch) return TT_FSI_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    return step(s, x_dev, labels_dev, target_dev, v_empty, B, loss_dev, true, st);
}

tt_fsi_status tt_fsi_student_predict(tt_fsi_student s, const float *x_dev, const float *target_dev, float v_empty,
                                     int B, float *phi_dev, struct CUstream_st *stream) {
    if (!s || !x_dev || !target_dev || !phi_dev || B < 1 || B > s->max_batch) return TT_FSI_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    tt_fsi_status r = forward(s, x_dev, B, false, st);
    if (r != TT_FSI_OK) return r;
    ttfsi_student::ProjectArgs p = project_args(s, target_dev, v_empty, B);
    p.phi = phi_dev;
    return chain(ttfsi_student::project_kernel, (unsigned)((B + kProjectRows - 1) / kProjectRows), 256, 0, st, p);
}

tt_fsi_status tt_fsi_student_get_state(tt_fsi_student s, float *params_host, float *adam_m_host, float *adam_v_host,
                                       int64_t *step) {
    if (!s) return TT_FSI_ERR_INVALID_ARG;
    const size_t bytes = (size_t)s->n_params * sizeof(float);
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess && params_host) e = cudaMemcpy(params_host, s->params, bytes, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && adam_m_host) e = cudaMemcpy(adam_m_host, s->m, bytes, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && adam_v_host) e = cudaMemcpy(adam_v_host, s->v, bytes, cudaMemcpyDeviceToHost);
    if (step) *step = s->step;
    return st_status(e);
}

tt_fsi_status tt_fsi_student_set_state(tt_fsi_student s, const float *params_host, const float *adam_m_host,
                                       const float *adam_v_host, int64_t step) {
    if (!s || step < 0) return TT_FSI_ERR_INVALID_ARG;
    const size_t bytes = (size_t)s->n_params * sizeof(float);
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess && params_host) e = cudaMemcpy(s->params, params_host, bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && adam_m_host) e = cudaMemcpy(s->m, adam_m_host, bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && adam_v_host) e = cudaMemcpy(s->v, adam_v_host, bytes, cudaMemcpyHostToDevice);
    s->step = step;
    tt_fsi_status r = st_status(e);
    if (r == TT_FSI_OK) r = refresh_bf16(s, nullptr);
    if (r == TT_FSI_OK) r = st_status(cudaDeviceSynchronize());
    return r;
}

tt_fsi_status tt_fsi_student_get_grads(tt_fsi_student s, float *grads_host) {
    if (!s || !grads_host) return TT_FSI_ERR_INVALID_ARG;
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess)
        e = cudaMemcpy(grads_host, s->grads, (size_t)s->n_params * sizeof(float), cudaMemcpyDeviceToHost);
    return st_status(e);
}

tt_fsi_status tt_fsi_student_check(tt_fsi_student s, struct CUstream_st *stream) {
    if (!s) return TT_FSI_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int h = 0;
    cudaError_t e = cudaMemcpyAsync(&h, s->err, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->err, 0, sizeof(int), st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return st_status(e);
    return h ? TT_FSI_ERR_TIMEOUT : TT_FSI_OK;
}

tt_fsi_status tt_fsi_surrogate_residual(const float *phi_dev, int B, int n_out, const unsigned *score_masks_dev,
                                        const unsigned *coal_dev, const float *vcoal_dev, int K, float *resid_dev,
                                        struct CUstream_st *stream) {
    if (B < 0 || n_out < 1 || K < 1) return TT_FSI_ERR_INVALID_ARG;
    if (B == 0) return TT_FSI_OK;
    if (!phi_dev || !score_masks_dev || !coal_dev || !vcoal_dev || !resid_dev) return TT_FSI_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    ttfsi_student::residual_kernel<<<(B + 7) / 8, 256, 0, st>>>(phi_dev, B, n_out, score_masks_dev, coal_dev, vcoal_dev,
                                                              K, resid_dev);
    return st_status(cudaGetLastError());
}

}  // extern "C"
