// Learned-proposal network: a small MLP trained on simulator output.
//
// Layers d0 -> d1 -> ... -> dL with ReLU between hidden layers and a linear
// output.  Weights are BF16 (an FP32 master copy is kept for the optimiser);
// every product accumulates in FP32 on the fifth-generation tensor cores
// (tcgen05.mma kind::f16, BF16 x BF16 -> FP32 in tensor memory).  Activations
// are stored in BF16 between layers.
//
// Kernels: one generic strided GEMM with fused epilogues (bias, ReLU, ReLU
// mask of the backward pass, FP32 or BF16 output), a column-sum for bias
// gradients, and the Adam update.  The GEMM computes one 128 x 64 output tile
// per CTA of 256 threads: 64-wide K chunks of both operands go into K-major
// core-matrix images in four buffers, one thread issues four 128 x N x 16 MMAs
// per chunk and commits to the buffer's mbarrier; eight warps read the
// accumulator with tcgen05.ld (one output row per lane, half the columns each)
// and apply the epilogue with vector stores.  Operands that are contiguous
// along K are staged with 16-byte asynchronous copies three chunks ahead;
// operands contiguous along the rows (both of dW = dZ^T X) as 8 x 8 blocks,
// eight 16-byte loads a thread transposed in registers.  The GEMMs of this
// network are small (256 x 512 x 1024 at most), so each is the latency of its
// chunks: with synchronous staging, element gathers of transposed operands and
// one 128 x 128 tile per CTA a forward and backward pass of batch 256 took
// 519 us, now 144 us.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

#include "../../include/mdx.h"
#include "mdx_internal.h"
#include "mdx_tc.cuh"

namespace mdx {

namespace {

constexpr int TBM = 128, TBN = 64, TBK = 64;    // output tile, K chunk (BF16 elements)
constexpr int kGemmThreads = 256;                // first half stages A, second half B
constexpr int kGemmStages = 4;
constexpr int kABytes = TBM * TBK * 2, kBBytes = TBN * TBK * 2;   // operand chunk images
constexpr long long kGemmWait = 1LL << 24;

enum : int { EPI_NONE = 0, EPI_BIAS = 1, EPI_RELU = 2, EPI_MASK = 4, EPI_BF16 = 8 };

struct GemmArgs {
    int M, N, K;
    const uint16_t *A;             // element (m, k) at A[m * sAm + k * sAk]  (BF16 bits)
    long long sAm, sAk;
    const uint16_t *B;             // element (k, n) at B[k * sBk + n * sBn]
    long long sBk, sBn;
    void *C;                       // element (m, n) at C[m * ldc + n] (FP32 or BF16)
    long long ldc;
    const float *bias;             // [N]
    const uint16_t *mask;          // BF16 [M][ldm]: keep where mask > 0 (ReLU derivative)
    long long ldm;
    int epi;
};

__device__ __forceinline__ uint16_t f2bf(float x) {
    return __bfloat16_as_ushort(__float2bfloat16_rn(x));
}

__device__ __forceinline__ float bf2f(uint16_t x) { return __bfloat162float(__ushort_as_bfloat16(x)); }

// Instruction descriptor of kind::f16 with BF16 A and B (both K-major) and an
// FP32 accumulator, shape M x N.
__device__ __forceinline__ uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16_tc(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}

// 16-byte asynchronous copy of which the first `bytes` are read, the rest zero.
__device__ __forceinline__ void copy16(uint16_t *dst, const uint16_t *src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::su32(dst)), "l"(src),
                 "r"(bytes)
                 : "memory");
}

// Transposes an 8 x 8 block of 16-bit elements held as eight rows of four words.
__device__ __forceinline__ void transpose8(uint4 (&v)[8]) {
    uint32_t w[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i][0] = v[i].x, w[i][1] = v[i].y, w[i][2] = v[i].z, w[i][3] = v[i].w;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        uint32_t o[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
            o[c] = __byte_perm(w[2 * c][r >> 1], w[2 * c + 1][r >> 1], (r & 1) ? 0x7632 : 0x5410);
        v[r] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// Stages ROWS rows from row0 (valid below `rows`) and K columns k0 .. k0+63
// (valid below K) of a strided BF16 matrix, element (r, k) at
// src[r * s_r + k * s_k], into a K-major core-matrix image: 16-byte units of
// 8 K-adjacent elements, 8-row groups 8 units (1024 bytes) apart.  t: thread
// 0..127 of the operand's half of the CTA.
template <int ROWS>
__device__ __forceinline__ void stage_operand(uint16_t *img, const uint16_t *src, long long s_r,
                                              long long s_k, int row0, int rows, int k0, int K, int t) {
    const bool al = (reinterpret_cast<uintptr_t>(src) & 15) == 0;
    if (s_k == 1 && (s_r & 7) == 0 && al) {
        // K contiguous: 8 units of one row are 128 contiguous bytes
#pragma unroll
        for (int u = 0; u < ROWS * 8 / 128; ++u) {
            const int i = t + 128 * u, r = i >> 3, kg = i & 7;
            const int row = row0 + r, k = k0 + kg * 8;
            const int bytes = row < rows ? max(0, min(16, 2 * (K - k))) : 0;
            copy16(img + (((r >> 3) * 8 + kg) * 64 + (r & 7) * 8),
                   bytes ? src + (long long)row * s_r + k : src, bytes);
        }
    } else if (s_r == 1 && (s_k & 7) == 0 && al) {
        // rows contiguous: thread = one 8-row x 8-K block (kg fixed per quarter-warp pass)
        for (int i = t; i < ROWS; i += 128) {
            const int rg = i % (ROWS / 8), kg = i / (ROWS / 8);
            const int row = row0 + rg * 8, k = k0 + kg * 8;
            uint4 v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                v[e] = make_uint4(0u, 0u, 0u, 0u);
                if (k + e < K) {
                    const uint16_t *p = src + (long long)(k + e) * s_k + row;
                    if (row + 8 <= rows) {
                        v[e] = __ldg(reinterpret_cast<const uint4 *>(p));
                    } else if (row < rows) {
                        alignas(16) uint16_t x[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) x[q] = row + q < rows ? p[q] : 0;
                        v[e] = *reinterpret_cast<const uint4 *>(x);
                    }
                }
            }
            transpose8(v);
#pragma unroll
            for (int e = 0; e < 8; ++e)
                *reinterpret_cast<uint4 *>(img + ((rg * 8 + kg) * 64 + e * 8)) = v[e];
        }
    } else {
        // any strides (narrow or unaligned operands)
        for (int i = t; i < ROWS * 8; i += 128) {
            const int r = i % ROWS, kg = i / ROWS;
            const int row = row0 + r, k = k0 + kg * 8;
            alignas(16) uint16_t x[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                x[e] = (row < rows && k + e < K) ? src[(long long)row * s_r + (long long)(k + e) * s_k] : 0;
            *reinterpret_cast<uint4 *>(img + (((r >> 3) * 8 + kg) * 64 + (r & 7) * 8)) =
                *reinterpret_cast<const uint4 *>(x);
        }
    }
}

// One launch: up to two independent GEMMs (of one layer's backward pass) and a
// column sum, in consecutive block ranges.
struct LayerArgs {
    GemmArgs g[2];
    int nx[2], tiles[2];           // output tiles along N, in all
    const uint16_t *dz;            // column sum: db[n] = sum_m dz[m][n] (null: none)
    int M, N;
    float *db;
};

struct GemmCtrl {
    uint64_t bar[kGemmStages];
    uint32_t tmem;
    int fail;                // first chunk after which a wait ran out
};

}  // namespace

// db[n] = sum_m dz[m][n] (dz BF16 [M][N]), FP32 accumulation: 32 columns a CTA,
// eight threads a column with every eighth row each (one thread per column
// walked 256 rows in 13 us), their parts added in order.
constexpr int kSumRows = kGemmThreads / 32;
__device__ void col_sum(const uint16_t *dz, int M, int N, float *db, int block) {
    __shared__ float part[kSumRows][32];
    const int c = threadIdx.x & 31, r = threadIdx.x >> 5, n = block * 32 + c;
    float s = 0.f;
    if (n < N) {
#pragma unroll 8
        for (int m = r; m < M; m += kSumRows) s += bf2f(dz[(long long)m * N + n]);
    }
    part[r][c] = s;
    __syncthreads();
    if (r == 0 && n < N) {
#pragma unroll
        for (int q = 1; q < kSumRows; ++q) s += part[q][c];
        db[n] = s;
    }
}

__global__ void __launch_bounds__(kGemmThreads) mlp_gemm_kernel(const __grid_constant__ LayerArgs A) {
    using namespace tc;
    int blk = blockIdx.x;
    if (blk >= A.tiles[0] + A.tiles[1]) {
        col_sum(A.dz, A.M, A.N, A.db, blk - A.tiles[0] - A.tiles[1]);
        return;
    }
    const int which = blk >= A.tiles[0] ? 1 : 0;
    const GemmArgs &g = A.g[which];
    if (which) blk -= A.tiles[0];
    extern __shared__ __align__(1024) unsigned char gsm[];
    GemmCtrl &C = *reinterpret_cast<GemmCtrl *>(gsm);
    unsigned char *img = gsm + 1024;              // [kGemmStages][A 16 KB, B 8 KB]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blk / A.nx[which] * TBM, n0 = blk % A.nx[which] * TBN;
    const int nvalid = min(TBN, g.N - n0);
    const int NT = (nvalid + 15) & ~15;                         // MMA N (multiple of 16)
    const int chunks = (g.K + TBK - 1) / TBK;
    if (tid == 0) {
        for (int b = 0; b < kGemmStages; ++b) bar_init(&C.bar[b], 1);
        C.fail = chunks;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 64;" ::"r"(
                         su32(&C.tmem))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    auto stage = [&](int c) {
        unsigned char *p = img + (size_t)(c % kGemmStages) * (kABytes + kBBytes);
        if (tid < 128)
            stage_operand<TBM>(reinterpret_cast<uint16_t *>(p), g.A, g.sAm, g.sAk, m0, g.M, c * TBK,
                               g.K, tid);
        else
            stage_operand<TBN>(reinterpret_cast<uint16_t *>(p + kABytes), g.B, g.sBn, g.sBk, n0, g.N,
                               c * TBK, g.K, tid - 128);
    };
    // one copy group per chunk, empty ones past the end
    auto stage_group = [&](int c) {
        if (c < chunks) stage(c);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int c = 0; c < kGemmStages - 1; ++c) stage_group(c);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = C.tmem;
    const uint32_t idesc = idesc_bf16(TBM, NT);
    bool ok = true;
    int committed = 0;   // chunks whose MMAs thread 0 has committed
    // waits until the MMAs of chunk c have read their buffer
    auto mma_wait = [&](int c) {
        long long i = 0;
        while (!bar_try(&C.bar[c % kGemmStages], (uint32_t)((c / kGemmStages) & 1)) && ++i < kGemmWait) {
        }
        return i < kGemmWait;
    };
    for (int c = 0; c < chunks; ++c) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kGemmStages - 2) : "memory");
        fence_async_smem();
        tc_fence_before();
        __syncthreads();
        // (a failure counts behind the next barrier, where every thread reads it)
        if (C.fail < c) {
            ok = false;
            break;
        }
        if (tid == 0) {
            tc_fence_after();
            const uint32_t a0 = su32(img) + (uint32_t)(c % kGemmStages) * (kABytes + kBBytes);
            const uint32_t b0 = a0 + kABytes;
#pragma unroll
            for (int kk = 0; kk < TBK / 16; ++kk) {
                const uint64_t ad = smem_desc(a0 + kk * 256u, 128u, 1024u);
                const uint64_t bd = smem_desc(b0 + kk * 256u, 128u, 1024u);
                mma_bf16_tc(tmem, ad, bd, idesc, (c | kk) ? 1u : 0u);
            }
            mma_commit(&C.bar[c % kGemmStages]);
            ++committed;
        }
        // the buffer of chunk c + 3 was read by chunk c - 1
        if (c + kGemmStages - 1 < chunks && c >= 1 && !mma_wait(c - 1))
            atomicMin(&C.fail, c);
        else
            stage_group(c + kGemmStages - 1);
    }
    // the last commit covers every MMA issued before it
    if (ok && chunks > 0) ok = mma_wait(chunks - 1);
    tc_fence_after();
    // epilogue: lane quarter warp % 4 (output rows), column half warp / 4
    const int m = m0 + (warp & 3) * 32 + lane;
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
    const bool vec32 = (g.ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(g.C) & 15) == 0;
    const bool vec16 = (g.ldc & 7) == 0 && (reinterpret_cast<uintptr_t>(g.C) & 15) == 0;
    const bool vecm = (g.ldm & 7) == 0 && (reinterpret_cast<uintptr_t>(g.mask) & 15) == 0;
    for (int cb = 16 * (warp >> 2); cb < NT; cb += 32) {
        float v[16];
        if (chunks > 0) {
            tmem_ld16(tmem + lane_base + (uint32_t)cb, v);
        } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = 0.f;
        }
        if (m >= g.M) continue;
        const bool full = cb + 16 <= nvalid;
        alignas(16) uint16_t mk[16];
        if (g.epi & EPI_MASK) {
            const uint16_t *mp = g.mask + (long long)m * g.ldm + n0 + cb;
            if (full && vecm) {
                *reinterpret_cast<uint4 *>(mk) = *reinterpret_cast<const uint4 *>(mp);
                *reinterpret_cast<uint4 *>(mk + 8) = *reinterpret_cast<const uint4 *>(mp + 8);
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) mk[j] = cb + j < nvalid ? mp[j] : 0;
            }
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            if (cb + j >= nvalid) break;
            float x = ok ? v[j] : __int_as_float(0x7fc00000);
            if (g.epi & EPI_BIAS) x += g.bias[n0 + cb + j];
            if (g.epi & EPI_RELU) x = fmaxf(x, 0.f);
            if ((g.epi & EPI_MASK) && !(bf2f(mk[j]) > 0.f)) x = 0.f;
            v[j] = x;
        }
        if (g.epi & EPI_BF16) {
            uint16_t *Cp = static_cast<uint16_t *>(g.C) + (long long)m * g.ldc + n0 + cb;
            alignas(16) uint16_t h[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) h[j] = f2bf(v[j]);
            if (full && vec16) {
                *reinterpret_cast<uint4 *>(Cp) = *reinterpret_cast<const uint4 *>(h);
                *reinterpret_cast<uint4 *>(Cp + 8) = *reinterpret_cast<const uint4 *>(h + 8);
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (cb + j < nvalid) Cp[j] = h[j];
            }
        } else {
            float *Cp = static_cast<float *>(g.C) + (long long)m * g.ldc + n0 + cb;
            if (full && vec32) {
#pragma unroll
                for (int j = 0; j < 16; j += 4)
                    *reinterpret_cast<float4 *>(Cp + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (cb + j < nvalid) Cp[j] = v[j];
            }
        }
    }
    if (!ok) {
        // a wait ran out: the copies and the MMAs in flight finish before the memory
        // is released (the last commit on each buffer's barrier)
        asm volatile("cp.async.wait_all;" ::: "memory");
        for (int bb = 0; tid == 0 && bb < kGemmStages; ++bb) {
            const int cnt = (committed + kGemmStages - 1 - bb) / kGemmStages;
            if (cnt <= 0) continue;
            long long i = 0;
            while (!bar_try(&C.bar[bb], (uint32_t)((cnt - 1) & 1)) && ++i < kGemmWait) {
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 64;" ::"r"(tmem) : "memory");
}

namespace {

constexpr size_t kGemmSmem = 1024 + kGemmStages * (size_t)(kABytes + kBBytes);
std::once_flag g_gemm_attr;

}  // namespace

// Launches the GEMMs g0 (and g1, may be null) and the column sum of dz into db.
static cudaError_t layer(const GemmArgs *g0, const GemmArgs *g1, const uint16_t *dz, int M, int N,
                         float *db, cudaStream_t s) {
    std::call_once(g_gemm_attr, [] {
        cudaFuncSetAttribute(mlp_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kGemmSmem);
    });
    LayerArgs A{};
    const GemmArgs *gs[2] = {g0, g1};
    for (int i = 0; i < 2; ++i) {
        A.nx[i] = 1;
        if (!gs[i] || gs[i]->M <= 0 || gs[i]->N <= 0) continue;
        A.g[i] = *gs[i];
        A.nx[i] = (gs[i]->N + TBN - 1) / TBN;
        A.tiles[i] = A.nx[i] * ((gs[i]->M + TBM - 1) / TBM);
    }
    A.dz = dz;
    A.M = M;
    A.N = N;
    A.db = db;
    const int blocks = A.tiles[0] + A.tiles[1] + (dz ? (N + 31) / 32 : 0);
    if (blocks == 0) return cudaSuccess;
    mlp_gemm_kernel<<<blocks, kGemmThreads, kGemmSmem, s>>>(A);
    return cudaGetLastError();
}

__global__ void f32_to_bf16_kernel(const float *x, long long n, uint16_t *y) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < n) y[i] = f2bf(x[i]);
}

// Adam (Kingma & Ba): m = b1 m + (1-b1) g, v = b2 v + (1-b2) g^2,
// w -= lr * (m / (1-b1^t)) / (sqrt(v / (1-b2^t)) + eps); BF16 copy refreshed.
__global__ void adam_kernel(long long n, float *w, uint16_t *wb, const float *g, float *m, float *v,
                            float lr, float b1, float b2, float eps, float c1, float c2) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    if (wb) wb[i] = f2bf(wi);
}

}  // namespace mdx

using namespace mdx;

static int mlp_check(const mdx_mlp *net, int batch) {
    if (!net || net->n_layers < 1 || net->n_layers > MDX_MLP_MAX_LAYERS)
        return set_last_error(MDX_ERR_ARG, "n_layers must be in 1..MDX_MLP_MAX_LAYERS");
    if (batch < 1) return set_last_error(MDX_ERR_ARG, "batch must be >= 1");
    for (int l = 0; l <= net->n_layers; ++l)
        if (net->dims[l] < 1) return set_last_error(MDX_ERR_ARG, "layer widths must be >= 1");
    for (int l = 0; l < net->n_layers; ++l)
        if (!net->W[l] || !net->b[l]) return set_last_error(MDX_ERR_ARG, "missing weights or biases");
    return MDX_OK;
}

static long long act_offset(const mdx_mlp *net, int batch, int l) {
    // activations of hidden layers 1..L-1, each [batch][d_l], concatenated
    long long off = 0;
    for (int j = 1; j < l; ++j) off += (long long)batch * net->dims[j];
    return off;
}

extern "C" size_t mdx_mlp_act_elems(const mdx_mlp *net, int batch) {
    if (mlp_check(net, batch)) return 0;
    return (size_t)act_offset(net, batch, net->n_layers);
}

extern "C" int mdx_mlp_forward(const mdx_mlp *net, int batch, const uint16_t *x, uint16_t *acts,
                               float *y, void *stream) {
    int rc = mlp_check(net, batch);
    if (rc) return rc;
    if (!x || !y || (net->n_layers > 1 && !acts)) return set_last_error(MDX_ERR_ARG, "null buffer");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const uint16_t *in = x;
    for (int l = 0; l < net->n_layers; ++l) {
        const int K = net->dims[l], N = net->dims[l + 1];
        const bool last = l == net->n_layers - 1;
        GemmArgs g{};
        g.M = batch;
        g.N = N;
        g.K = K;
        g.A = in;
        g.sAm = K;
        g.sAk = 1;
        g.B = net->W[l];        // W[n][k] -> B(k, n) = W[n * K + k]
        g.sBk = 1;
        g.sBn = K;
        g.bias = net->b[l];
        if (last) {
            g.C = y;
            g.ldc = N;
            g.epi = EPI_BIAS;
        } else {
            uint16_t *out = acts + act_offset(net, batch, l + 1);
            g.C = out;
            g.ldc = N;
            g.epi = EPI_BIAS | EPI_RELU | EPI_BF16;
            in = out;
        }
        if (layer(&g, nullptr, nullptr, 0, 0, nullptr, s) != cudaSuccess)
            return set_last_error(MDX_ERR_CUDA, "mlp forward launch failed");
    }
    return MDX_OK;
}

extern "C" size_t mdx_mlp_work_elems(const mdx_mlp *net, int batch) {
    if (mlp_check(net, batch)) return 0;
    int dmax = 0;
    for (int l = 0; l <= net->n_layers; ++l) dmax = net->dims[l] > dmax ? net->dims[l] : dmax;
    return (size_t)2 * batch * dmax;
}

extern "C" int mdx_mlp_backward(const mdx_mlp *net, int batch, const uint16_t *x,
                                const uint16_t *acts, const float *dy, float *const *dW,
                                float *const *db, uint16_t *work, void *stream) {
    int rc = mlp_check(net, batch);
    if (rc) return rc;
    if (!x || !dy || !dW || !db || !work) return set_last_error(MDX_ERR_ARG, "null buffer");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int dmax = 0;
    for (int l = 0; l <= net->n_layers; ++l) dmax = net->dims[l] > dmax ? net->dims[l] : dmax;
    uint16_t *dz = work;                              // BF16 [batch][d_{l+1}] of the current layer
    uint16_t *dz_next = work + (long long)batch * dmax;
    // output layer: dz = dy (linear), rounded to BF16 once
    {
        const long long n = (long long)batch * net->dims[net->n_layers];
        f32_to_bf16_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(dy, n, dz);
    }
    for (int l = net->n_layers - 1; l >= 0; --l) {
        const int K = net->dims[l], N = net->dims[l + 1];
        const uint16_t *in = (l == 0) ? x : acts + act_offset(net, batch, l);
        // dW[n][k] = sum_m dz[m][n] in[m][k]
        GemmArgs g{};
        g.M = N;
        g.N = K;
        g.K = batch;
        g.A = dz;               // A(n, m) = dz[m * N + n]
        g.sAm = 1;
        g.sAk = N;
        g.B = in;               // B(m, k) = in[m * K + k]
        g.sBk = K;
        g.sBn = 1;
        g.C = dW[l];
        g.ldc = K;
        g.epi = EPI_NONE;
        // dz_prev[m][k] = (sum_n dz[m][n] W[n][k]) * [act_l[m][k] > 0], BF16
        GemmArgs h{};
        if (l > 0) {
            h.M = batch;
            h.N = K;
            h.K = N;
            h.A = dz;
            h.sAm = N;
            h.sAk = 1;
            h.B = net->W[l];    // B(n, k) = W[n * K + k]
            h.sBk = K;
            h.sBn = 1;
            h.C = dz_next;
            h.ldc = K;
            h.mask = in;
            h.ldm = K;
            h.epi = EPI_MASK | EPI_BF16;
        }
        // dW, dz_prev and db of a layer need only dz: one launch
        if (layer(&g, l > 0 ? &h : nullptr, dz, batch, N, db[l], s) != cudaSuccess)
            return set_last_error(MDX_ERR_CUDA, "mlp backward launch failed");
        uint16_t *t = dz;
        dz = dz_next;
        dz_next = t;
    }
    if (cudaGetLastError() != cudaSuccess) return set_last_error(MDX_ERR_CUDA, "mlp backward launch failed");
    return MDX_OK;
}

extern "C" int mdx_adam_step(long long n, float *w, uint16_t *w_bf16, const float *g, float *m,
                             float *v, float lr, float beta1, float beta2, float eps, int t,
                             void *stream) {
    if (n < 0 || !w || !g || !m || !v || t < 1) return set_last_error(MDX_ERR_ARG, "bad Adam arguments");
    if (n == 0) return MDX_OK;
    const float c1 = 1.f - powf(beta1, (float)t), c2 = 1.f - powf(beta2, (float)t);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    adam_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, w, w_bf16, g, m, v, lr, beta1, beta2,
                                                            eps, c1, c2);
    if (cudaGetLastError() != cudaSuccess) return set_last_error(MDX_ERR_CUDA, "adam launch failed");
    return MDX_OK;
}

extern "C" int mdx_f32_to_bf16(long long n, const float *x, uint16_t *y, void *stream) {
    if (n < 0 || (n > 0 && (!x || !y))) return set_last_error(MDX_ERR_ARG, "bad conversion arguments");
    if (n == 0) return MDX_OK;
    f32_to_bf16_kernel<<<(unsigned)((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(x, n, y);
    if (cudaGetLastError() != cudaSuccess) return set_last_error(MDX_ERR_CUDA, "conversion launch failed");
    return MDX_OK;
}
