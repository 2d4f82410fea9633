// Small von Karman plates with many stress modes (at most 32 transverse and 129 to
// 256 stress modes): the forward pass with the coupling rows in registers.
//
// The resident kernel (mdx_resident.cu) takes one warp per stress mode, eight a
// CTA, so at most 128 of them on the 16 CTAs of a cluster.  Here a stress mode is
// one warp of a CTA of up to 16, each lane holding one row of H^k:
//   * one cluster of cs CTAs per plate; CTA r owns the stress modes
//     k = r nkc .. r nkc + nkc - 1, one warp each, lane i the row of the
//     class-ordered mode i (columns of class a ^ class(k), the only nonzero block);
//   * u_i = H^k_i q_b from the class-ordered q in shared memory, eta_k a warp sum;
//   * the force terms kappa_k eta_k u_i go to a per-mode shared array
//     (double-buffered by step parity); after one cluster barrier, thread m of
//     every CTA gathers f_m from all CTAs over distributed shared memory in a
//     fixed order, so every CTA applies the identical update to all modes.
// Bound: the dependent loads of that gather and the cluster barrier.  Forward pass
// of 1 000 steps, streaming kernel and here: 30 x 130 modes 22.2 and 7.6 ms, 32 x 200
// 16.5 and 9.7 ms, 16 x 240 20.8 and 10.8 ms.  The hardware cluster barrier needs no spin loop:
// every CTA of a cluster is resident, and all run the same number of steps.
#include <cuda_runtime.h>

#include "../../include/mdx.h"
#include "mdx_common.cuh"

namespace mdx {

namespace {

constexpr int kEChunk = 256;   // excitation samples staged per shared-memory block

__device__ __forceinline__ uint32_t cta_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
                 "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Load a float from the shared memory of CTA `rank` of this cluster at the
// address that `local` has in this CTA.
__device__ __forceinline__ float ld_peer(const float *local, uint32_t rank) {
    const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(local));
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(ra) : "memory");
    return v;
}

__device__ __forceinline__ int pick4c(const int (&v)[4], int a) {
    return a == 0 ? v[0] : (a == 1 ? v[1] : (a == 2 ? v[2] : v[3]));
}

__device__ __forceinline__ int class_of(const InstDesc &d, int i) {
    return (i >= d.ocls[1]) + (i >= d.ocls[2]) + (i >= d.ocls[3]);
}

}  // namespace

__global__ void __launch_bounds__(32 * kClusterMaxNkc, 1) cluster_kernel(const ClusterParams P) {
    constexpr int RL = kClusterMaxModes;
    __shared__ __align__(16) float qc[4 * RL];                  // class blocks of q (padded)
    __shared__ float fslot[2][kClusterMaxNkc][RL];              // force terms
    __shared__ float ebuf[2 * kEChunk];                         // excitation
    const int cs = P.cs, nkc = P.nkc;
    const int nthreads = blockDim.x;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cta_rank();
    const int plate = P.plates[blockIdx.x / cs];
    const InstDesc d = P.inst[plate];
    const int N = d.N;
    const long long TM = P.total_modes;

    // ---- this thread's coupling row: stress slot, class-ordered row i
    const int kslot = warp, i = lane;
    const int kl = (int)rank * nkc + kslot;        // internal stress index
    float h[RL];
#pragma unroll
    for (int j = 0; j < RL; ++j) h[j] = 0.f;
    int qoff = 0;                                  // class block of the row's columns
    float kap = 0.f;
    int ia = 0, ip = 0;                            // row class and position in it
    if (kl < d.M && i < N) {
        const ClusterK K = P.kinfo[d.k_off + kl];
        ia = class_of(d, i);
        ip = i - pick4c(d.ocls, ia);
        const int b = ia ^ K.c;
        const int nbc = pick4c(d.ncls, b);
        long long sb = 0;
        for (int a2 = 0; a2 < ia; ++a2)
            sb += (long long)pick4c(d.ncls, a2) * K.mc * ((pick4c(d.ncls, a2 ^ K.c) + 3) & ~3);
        const float *row = P.H + K.off + sb + ((long long)ip * K.mc + K.kpos) * ((nbc + 3) & ~3);
#pragma unroll
        for (int j = 0; j < RL; ++j) h[j] = (j < nbc) ? row[j] : 0.f;
        qoff = b * RL;
        kap = P.kappa[d.k_off + kl];
    } else if (i < N) {
        ia = class_of(d, i);
        ip = i - pick4c(d.ocls, ia);
    }
    const bool row_live = i < N;

    // ---- per-mode state and coefficients: thread m < N owns class-ordered mode m
    float qhi = 0.f, qlo = 0.f, vhi = 0.f, vlo = 0.f;
    float eps = 0.f, rw2 = 0.f, rw2l = 0.f, r = 0.f, bw = 0.f, cw = 0.f, clo = 0.f;
    int ma = 0, mpos = 0;
    if (tid < N) {
        const long long m = d.mode_off + P.perm[d.perm_off + tid];
        qhi = P.state_io[m];
        qlo = P.state_io[TM + m];
        vhi = P.state_io[2 * TM + m];
        vlo = P.state_io[3 * TM + m];
        eps = P.coef.eps[m];
        rw2 = P.coef.rw2[m];
        rw2l = P.coef.rw2lo[m];
        r = P.coef.r[m];
        bw = P.coef.b[m];
        cw = P.coef.c[m];
        clo = P.coef.clo[m];
        ma = class_of(d, tid);
        mpos = tid - pick4c(d.ocls, ma);
    }
    for (int e = tid; e < 4 * RL; e += nthreads) qc[e] = 0.f;
    __syncthreads();
    if (tid < N) qc[ma * RL + mpos] = qhi;
    const float *exc = P.exc ? P.exc + (long long)plate * P.total_steps : nullptr;
    // every CTA of the cluster is running before any peer access
    cluster_sync_all();

    for (int it = 0; it < P.steps; ++it) {
        const int n = P.n_begin + it;
        const int buf = it & 1;
        if ((it % kEChunk) == 0) {
            float *eb = ebuf + ((it / kEChunk) & 1) * kEChunk;
            for (int e = tid; e < kEChunk; e += nthreads)
                eb[e] = (exc && it + e < P.steps) ? exc[n + e] : 0.f;
        }
        // u_i = H^k_i q_b, from registers and the class-blocked q
        float u = 0.f;
        {
            const float4 *q4 = reinterpret_cast<const float4 *>(qc + qoff);
            float u1 = 0.f;
#pragma unroll
            for (int j = 0; j < RL / 4; j += 2) {
                const float4 a = q4[j];
                u = fmaf(h[4 * j], a.x, u);
                u = fmaf(h[4 * j + 1], a.y, u);
                u = fmaf(h[4 * j + 2], a.z, u);
                u = fmaf(h[4 * j + 3], a.w, u);
                const float4 c = q4[j + 1];
                u1 = fmaf(h[4 * j + 4], c.x, u1);
                u1 = fmaf(h[4 * j + 5], c.y, u1);
                u1 = fmaf(h[4 * j + 6], c.z, u1);
                u1 = fmaf(h[4 * j + 7], c.w, u1);
            }
            u += u1;
        }
        const float qi = (i < N) ? qc[ia * RL + ip] : 0.f;
        const float part = warp_sum(row_live ? qi * u : 0.f);
        fslot[buf][kslot][i] = row_live ? kap * part * u : 0.f;
        cluster_sync_all();
        // f_m from every CTA's slots (same order in every CTA), then the update
        float ys = 0.f, ye = 0.f;
        if (tid < N) {
            float f = 0.f;
            for (int rr = 0; rr < cs; ++rr)
                for (int q = 0; q < nkc; ++q)
                    f += ld_peer(&fslot[buf][q][tid], (uint32_t)rr);
            const float e = ebuf[((it / kEChunk) & 1) * kEChunk + (it % kEChunk)];
            sv_step(qhi, qlo, vhi, vlo, eps, rw2, rw2l, r, fmaf(bw, e, -f));
            pickup_add(ys, ye, cw, clo, qhi, qlo);
            qc[ma * RL + mpos] = qhi;
        }
        if (warp == 0) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float s2 = __shfl_xor_sync(0xffffffffu, ys, o);
                const float e2 = __shfl_xor_sync(0xffffffffu, ye, o);
                pickup_merge(ys, ye, s2, e2);
            }
            if (rank == 0 && lane == 0) {
                const float y = ys + ye;
                if (P.audio) P.audio[(long long)plate * P.total_steps + n] = y;
                if (!isfinite(y)) set_status(P.status, plate, MDX_ERR_NONFINITE);
            }
        }
        __syncthreads();
    }
    if (rank == 0 && tid < N) {
        const long long m = d.mode_off + P.perm[d.perm_off + tid];
        P.state_io[m] = qhi;
        P.state_io[TM + m] = qlo;
        P.state_io[2 * TM + m] = vhi;
        P.state_io[3 * TM + m] = vlo;
    }
    // no CTA leaves while a peer may still read its shared memory
    cluster_sync_all();
}

static void cluster_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *at, int cs, int nkc,
                           int n_plates, cudaStream_t s) {
    cfg.gridDim = dim3((unsigned)(n_plates * cs));
    cfg.blockDim = dim3((unsigned)(32 * nkc));
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
}

cudaError_t launch_cluster(const ClusterParams &P, int n_plates, cudaStream_t s) {
    if (P.steps <= 0 || n_plates <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    cluster_config(cfg, at, P.cs, P.nkc, n_plates, s);
    return cudaLaunchKernelEx(&cfg, cluster_kernel, P);
}

// Allows clusters above the portable size where needed and reports how many
// clusters of this shape the device can hold at once (0: not launchable).  The
// attribute belongs to the kernel, not to a plan: it is only ever raised, so a
// plan with a portable cluster never withdraws it from another plan's larger one.
cudaError_t cluster_check(int cs, int nkc, int *max_clusters) {
    *max_clusters = 0;
    const void *fn = reinterpret_cast<const void *>(cluster_kernel);
    if (cs > 8) {
        const cudaError_t e =
            cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    cluster_config(cfg, at, cs, nkc, 1, nullptr);
    return cudaOccupancyMaxActiveClusters(max_clusters, fn, &cfg);
}

}  // namespace mdx
