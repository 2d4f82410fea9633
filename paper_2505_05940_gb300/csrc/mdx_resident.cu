// Resident von Karman plates: every pass of the time loop (forward, recompute,
// reverse and the fused sweep) with the coupling tensor held on the SMs for the
// whole launch.
//
// Per step and plate (Sec. 3.1, Eq. 9 with C^s_pn = H^n_ps; Sec. 3.2, Eq. 20),
// as in the streaming plate kernel: u^k = H^k q, eta_k = q . u^k,
// f = sum_k kappa_k eta_k u^k, then the difference-form update and the pickup;
// the reverse sweep adds z^k = H^k w, xi_k = w . u^k and
// J w = sum_k kappa_k (2 xi_k u^k + eta_k z^k), the fused sweep also the
// recompute of the previous segment (a third right-hand side).
//
// Why: streamed once per step, 64 plates of 200 x 50 modes move 128 MB per
// step and the pass was bound by the synchronisation of its stages (28.8 us
// forward, 40 us fused per step).  Plates are independent, so they need not
// advance together: one plate at a time fits a few SMs.  A plate runs on `sub`
// CTAs (1 to 16) of one thread-block cluster through the whole time loop;
// clusters that do not fit at once run one after the other.
//
// Rows: one warp per stress mode k.  Lanes 8 a .. 8 a + 7 hold the rows of
// class a (row l + 8 r of the class in lane l, register row r), whose only
// nonzero columns are those of class a ^ class(k), so all rows of a lane share
// their right-hand-side loads (four broadcast addresses a warp, one wavefront)
// and eta_k is a sum within the warp: no barrier before the forces.  A plate
// without classes (N <= 56) spreads its rows over the 32 lanes.  The rows live
// in registers (NREG rows) and in tensor memory (NTM rows), used as a
// thread-private extension of the register file.  Tensor memory rather than
// shared memory: reading 224 words a thread with their FMAs took 512 cycles
// per CTA of 256 threads (448 of them the FMAs), from shared memory (LDS.128)
// 1 800.  Products are packed FMAs (two columns at a time).
//
// Exchange: rank r owns the modes [N r / sub, N (r + 1) / sub).  After one CTA
// barrier every CTA adds its warps' forces and stores each mode's part into
// its owner's shared memory (st.async, completing on the owner's mbarrier); the
// owner adds the parts in rank order, updates its modes and stores the new
// right-hand sides into every peer the same way (its warps hold the state
// redundantly and serve different peers).  Sending every part to every peer
// instead needs one hop less but `sub` times the stores, which the SM-to-SM
// network takes at 13 cycles per warp store: 730 cycles a step for 8 CTAs of
// 200 modes (1 525 with three right-hand sides).
//
// A spare warp sums the pickups of eight steps at a time (forward and
// recompute), off the step's chain.
//
// Bound: the packed FMAs (two warps a scheduler) plus the latency of the
// dependent chain (one barrier, one warp reduction, two exchanges, the update).
#include <cuda_runtime.h>

#include <algorithm>

#include "../../include/mdx.h"
#include "mdx_common.cuh"
#include "mdx_tc.cuh"

namespace mdx {

namespace {

using namespace tc;

typedef unsigned long long u64;

constexpr int kResMaxWarps = 7;              // row warps of a CTA (and the spare warp)
constexpr int kPickSteps = 8;                // pickups reduced together by the spare warp
// Shared memory asked for per tensor-memory column: above 233 472 / 544, the SM's
// shared memory over one allocation step more than its 512 columns, so any CTAs
// that fit an SM by shared memory hold at most 512 columns together.
constexpr size_t kSmemPerColumn = 430;
constexpr size_t kResStatic = 1024;          // room for the static shared memory
constexpr long long kResWait = 1LL << 22;    // bound of every wait (polls)

__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
                 "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t peer_addr(uint32_t local, uint32_t rank) {
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local), "r"(rank));
    return ra;
}

// Remote stores that complete bytes on the receiver's mbarrier.
__device__ __forceinline__ void push1(uint32_t dst, uint32_t bar, float x) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::
                     "r"(dst), "r"(__float_as_uint(x)), "r"(bar) : "memory");
}
__device__ __forceinline__ void push2(uint32_t dst, uint32_t bar, float x, float y) {
    asm volatile(
        "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::
            "r"(dst), "r"(__float_as_uint(x)), "r"(__float_as_uint(y)), "r"(bar) : "memory");
}
__device__ __forceinline__ void push4(uint32_t dst, uint32_t bar, float x, float y, float z) {
    asm volatile(
        "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, "
        "[%5];" ::"r"(dst), "r"(__float_as_uint(x)), "r"(__float_as_uint(y)),
        "r"(__float_as_uint(z)), "r"(0), "r"(bar) : "memory");
}

__device__ __forceinline__ u64 ffma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 pack2(uint32_t lo, uint32_t hi) {
    return (u64)lo | ((u64)hi << 32);
}
__device__ __forceinline__ float sum2(u64 a) {
    return __uint_as_float((uint32_t)a) + __uint_as_float((uint32_t)(a >> 32));
}


__device__ __forceinline__ int pick4r(const int (&v)[4], int a) {
    return a == 0 ? v[0] : (a == 1 ? v[1] : (a == 2 ? v[2] : v[3]));
}

// Columns j .. j + 7 of two adjacent tensor-memory rows (16 words).
__device__ __forceinline__ void tmem_ld_rows2(uint32_t addr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
        "%12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(addr));
}
__device__ __forceinline__ void tmem_st8(uint32_t addr, const float (&v)[8]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr),
        "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
        "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
        "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7]))
        : "memory");
}
// The loaded words are operands of the wait, so no use of them moves above it.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                   "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                   "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]));
}

// Right-hand-side blocks: q (two copies in a reverse pass: the next step's is
// written while this one is read), w, q' of the recompute.
__host__ __device__ constexpr int rhs_blocks(int R) { return R == 1 ? 1 : R + 1; }

// Shared-memory layout (float offsets from the dynamic base), the same on the
// host.  W warps, kernel row length LM, N modes at most, NO owned modes at most.
struct ResLayout {
    int QB, PS;                 // strides: class block, pickup row
    int rhs, fp, xch, hs, coef, pick, gacc, vst, end;
};

__host__ __device__ inline ResLayout res_layout(int R, int W, int LM, int L, int N, int NO, int sub,
                                                int nsm) {
    ResLayout o;
    // class blocks 8 banks apart, so that the four classes' accesses do not collide
    o.QB = ((LM + 31) & ~31) + 8;
    o.PS = ((2 * N + 31) & ~31) + 8;
    int p = 16;                 // mbarriers, tensor-memory base
    o.rhs = p;                  // [blocks][4][QB]
    p += rhs_blocks(R) * 4 * o.QB;
    o.fp = p;                   // [W][R][4][QB] forces of each warp
    p += W * R * 4 * o.QB;
    o.xch = p;                  // [2][sub][NO] x (1, 2 or 4 floats): parts of the owned modes
    if (sub > 1) p += 2 * sub * NO * (R == 3 ? 4 : R);
    p = (p + 3) & ~3;
    o.hs = p;                   // [nsm][L / 4][32 W] x 4: coupling rows (thread-private)
    p += nsm * L * 32 * W;
    o.coef = p;                 // [7][32 W] coefficients of the updated modes
    p += 7 * 32 * W;
    o.pick = p;                 // [2][kPickSteps][PS] pickup terms
    if (R == 1) p += 2 * kPickSteps * o.PS;
    o.gacc = p;                 // [GA_N][2][32 W] gradient sums
    if (R >= 2) p += GA_N * 2 * 32 * W;
    o.vst = p;                  // [32 W] v^n of the next step
    if (R >= 2) p += 32 * W;
    o.end = p;
    return o;
}

// Asynchronous 4-byte copy from global to shared memory (no register holds the
// value, so nothing waits for it before copies_done).
__device__ __forceinline__ void copy4(float *dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(su32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Named barrier of n threads.
__device__ __forceinline__ void bar_sync_id(int id, int n) {
    __syncwarp();
    asm volatile("barrier.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive_id(int id, int n) {
    __syncwarp();
    asm volatile("barrier.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// One warp's products u[r][x] = sum_j H[r][j] q_x[j] over NTM tensor-memory
// rows ([column / 8][row][8], read two rows at a time, the next pair in flight
// during this pair's FMAs) and NSM shared-memory rows.  The loop over the
// columns stays rolled: unrolled with rows in registers the step's code, run
// once per step by a few warps, was bound by instruction fetch and spills.
template <int R, int NTM, int NSM>
__device__ __forceinline__ void row_products(const float4 *hs, int hs_stride, uint32_t taddr, int L,
                                             const float *const (&q)[R], float (&u)[NTM + NSM][R]) {
    constexpr int NA = NTM + NSM, NP = NTM / 2, UN = (NP & 1) ? 2 : 1;
    // few rows: two chains per row, the FMAs' latency is what bounds them
    constexpr int SP = NA <= 4 ? 2 : 1;
    static_assert(NTM > 0 && NTM % 2 == 0, "tensor-memory rows are read in pairs");
    u64 acc[NA][R][SP];
#pragma unroll
    for (int s = 0; s < NA; ++s)
#pragma unroll
        for (int x = 0; x < R; ++x)
#pragma unroll
            for (int p = 0; p < SP; ++p) acc[s][x][p] = 0ull;
    uint32_t tm[2][16];
    tmem_ld_rows2(taddr, tm[0]);
    const int row4 = (L / 4) * hs_stride;
#pragma unroll 1
    for (int j0 = 0; j0 < L; j0 += 8 * UN) {
#pragma unroll
        for (int h = 0; h < UN; ++h) {
            const int j = j0 + 8 * h;
            if (UN > 1 && j >= L) break;
            ulonglong2 qa[R], qb[R];
#pragma unroll
            for (int x = 0; x < R; ++x) {
                qa[x] = *reinterpret_cast<const ulonglong2 *>(q[x] + j);
                qb[x] = *reinterpret_cast<const ulonglong2 *>(q[x] + j + 4);
            }
            const float4 *hp = hs + (j / 4) * hs_stride;
            ulonglong2 ha[NSM > 0 ? NSM : 1], hb[NSM > 0 ? NSM : 1];
#pragma unroll
            for (int s = 0; s < NSM; ++s) {
                ha[s] = *reinterpret_cast<const ulonglong2 *>(hp + s * row4);
                hb[s] = *reinterpret_cast<const ulonglong2 *>(hp + s * row4 + hs_stride);
            }
#pragma unroll
            for (int g = 0; g < NP; ++g) {
                const int par = (h * NP + g) & 1;
                uint32_t (&w)[16] = tm[par];
                tmem_wait_ld(w);
                // beyond the last chunk the pair is read again and not used
                const bool more = g + 1 < NP || j + 8 < L;
                tmem_ld_rows2(taddr + (uint32_t)(more ? j * NTM + 16 * (g + 1) : 0), tm[par ^ 1]);
#pragma unroll
                for (int s = 0; s < 2; ++s)
#pragma unroll
                    for (int x = 0; x < R; ++x) {
                        u64 (&a)[SP] = acc[2 * g + s][x];
                        a[0] = ffma2(pack2(w[8 * s], w[8 * s + 1]), qa[x].x, a[0]);
                        a[SP - 1] = ffma2(pack2(w[8 * s + 2], w[8 * s + 3]), qa[x].y, a[SP - 1]);
                        a[0] = ffma2(pack2(w[8 * s + 4], w[8 * s + 5]), qb[x].x, a[0]);
                        a[SP - 1] = ffma2(pack2(w[8 * s + 6], w[8 * s + 7]), qb[x].y, a[SP - 1]);
                    }
            }
#pragma unroll
            for (int s = 0; s < NSM; ++s)
#pragma unroll
                for (int x = 0; x < R; ++x) {
                    u64 (&a)[SP] = acc[NTM + s][x];
                    a[0] = ffma2(ha[s].x, qa[x].x, a[0]);
                    a[SP - 1] = ffma2(ha[s].y, qa[x].y, a[SP - 1]);
                    a[0] = ffma2(hb[s].x, qb[x].x, a[0]);
                    a[SP - 1] = ffma2(hb[s].y, qb[x].y, a[SP - 1]);
                }
        }
    }
    tmem_wait_ld(tm[0]);
    tmem_wait_ld(tm[1]);
#pragma unroll
    for (int s = 0; s < NA; ++s)
#pragma unroll
        for (int x = 0; x < R; ++x)
            u[s][x] = SP == 2 ? sum2(acc[s][x][0]) + sum2(acc[s][x][SP - 1]) : sum2(acc[s][x][0]);
}

}  // namespace

template <int R, int NTM, int NSM, int LMAX>
__global__ void __launch_bounds__(256, 1) resident_kernel(const ResidentParams Q) {
    extern __shared__ __align__(16) float sm[];
    __shared__ ResCta A;
    __shared__ InstDesc d;
    const PlateParams &P = Q.p;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr bool REV = R >= 2, FWD = R == 1, FUSED = R == 3;
    constexpr int NR = NTM + NSM;                 // rows of a lane
    constexpr int XF = R == 3 ? 4 : R;            // floats per exchanged entry
    constexpr int QB = ((LMAX + 31) & ~31) + 8;
    const int W = Q.warps, WT = 32 * W;
    const ResLayout O = res_layout(R, W, LMAX, Q.L, Q.n_max, Q.no_max, Q.max_sub, NSM);
    uint64_t *bar_f = reinterpret_cast<uint64_t *>(sm);        // forces of the owned modes
    uint64_t *bar_q = bar_f + 1;                               // new right-hand sides
    uint64_t *bar_y = bar_f + 2;                               // pickup terms (two buffers)
    uint32_t *tbase = reinterpret_cast<uint32_t *>(sm + 8);
    const long long TM = P.total_modes;
    for (int e = tid; e < (int)(sizeof(ResCta) / 4); e += blockDim.x)
        reinterpret_cast<int *>(&A)[e] = reinterpret_cast<const int *>(Q.ctas + blockIdx.x)[e];
    for (int e = 16 + tid; e < O.end; e += blockDim.x) sm[e] = 0.f;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         su32(tbase)), "r"(Q.tcols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem0 = *tbase;
    const bool used = A.plate >= 0;
    for (int e = tid; used && e < (int)(sizeof(InstDesc) / 4); e += blockDim.x)
        reinterpret_cast<int *>(&d)[e] = reinterpret_cast<const int *>(P.inst + A.plate)[e];
    __syncthreads();

    const int N = used ? d.N : 0, nk = A.nk, sub = max(A.sub, 1), rank = A.rank, L = A.L;
    const bool cls = used && d.parity;
    const int m0 = (int)((long long)N * rank / sub);
    const int no = (int)((long long)N * (rank + 1) / sub) - m0;   // owned modes
    const int C = max((no + 31) / 32, 1);         // chunks of 32 owned modes
    if (tid == 0) {
        bar_init(bar_f, 1);
        bar_init(bar_q, sub > 1 ? 1 : C);
        bar_init(bar_y, 1);
        bar_init(bar_y + 1, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (sub > 1) {
            bar_expect_tx(bar_f, (uint32_t)(sub * no * XF * 4));
            bar_expect_tx(bar_q, (uint32_t)(N * 4 * (FUSED ? 2 : 1)));
        }
    }
    // class row of a user-order mode, and its place in a right-hand-side block
    auto class_pos = [&](int i) {
        if (!cls) return i;
        const int row = Q.iperm[d.perm_off + i];
        const int a = (row >= d.ocls[1]) + (row >= d.ocls[2]) + (row >= d.ocls[3]);
        return a * QB + row - pick4r(d.ocls, a);
    };
    float *const rhs = sm + O.rhs;
    constexpr int bw = 2 * 4 * QB, br = 3 * 4 * QB;   // blocks: q (twice in reverse), w, q'
    const int rsteps = FUSED ? P.rev_steps : P.steps;
    const float *rec0 = P.state_io;                            // incoming forward state
    if (FUSED) rec0 = P.ckpt + (long long)(P.rec_begin / P.ckpt_K) * kStateArrays * TM;
    else if (FWD && P.mode == MODE_RECOMPUTE)
        rec0 = P.ckpt + (long long)(P.n_begin / P.ckpt_K) * kStateArrays * TM;
    // this thread's share of the plate's modes (two at most): place, owner's slot
    // and barrier; the first step's right-hand sides
    int mp[2] = {0, 0};
    uint32_t mdst[2] = {0u, 0u}, mbar[2] = {0u, 0u};
    bool mon[2] = {false, false};
    if (used && tid < WT) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = tid + h * WT;
            if (i >= N) continue;
            mon[h] = true;
            const long long m = d.mode_off + i;
            mp[h] = class_pos(i);
            if (sub > 1) {
                const int own = ((i + 1) * sub - 1) / N;
                const int o0 = (int)((long long)N * own / sub);
                mdst[h] = peer_addr(su32(sm + O.xch) + (uint32_t)((rank * Q.no_max + i - o0) * XF * 4),
                                    (uint32_t)(A.base + own));
                mbar[h] = peer_addr(su32(bar_f), (uint32_t)(A.base + own));
            }
            if (FWD) rhs[mp[h]] = rec0[m];
            if (REV) {
                rhs[mp[h]] = P.seg_q[(long long)(rsteps - 1) * TM + m];
                rhs[bw + mp[h]] = P.coef.r[m] * P.adj[m];
            }
            if (FUSED) rhs[br + mp[h]] = rec0[m];
        }
    }
    __syncthreads();
    cluster_sync_all();      // every peer's barriers exist before the first store

    const bool pick_here = FWD && used && rank == sub - 1;
    if (used && tid < WT) {
        // ---- row role: rows of stress mode k0 + warp
        const bool kon = warp < nk;
        const int ra = cls ? lane >> 3 : 0;
        const int gl = cls ? 8 : 32, l0 = cls ? lane & 7 : lane;
        const int kl = A.k0 + warp;
        int kc = 0;
        const uint32_t taddr = tmem0 + ((uint32_t)(32 * (warp & 3)) << 16) +
                               (warp >= 4 ? (uint32_t)(Q.tcols / 2) : 0u);
        float4 *const hsm = reinterpret_cast<float4 *>(sm + O.hs) + tid;
        float kap = 0.f, ks = 0.f, kcmp = 0.f;                  // kappa, d kappa (Kahan)
        {
            const int ncl = cls ? pick4r(d.ncls, ra) : N;       // rows of this lane's class
            long long off = 0;
            int n = 0, stride = 0;
            if (kon) {
                kap = P.kappa[d.k_off + kl];
                if (REV) {
                    ks = P.kacc[2 * (d.k_off + kl)];
                    kcmp = P.kacc[2 * (d.k_off + kl) + 1];
                }
                if (cls) {
                    const ClusterK K = Q.kinfo[d.k_off + kl];
                    kc = K.c;
                    n = pick4r(d.ncls, ra ^ kc);
                    const int w = (n + 3) & ~3;
                    long long sb = 0;
                    for (int a2 = 0; a2 < ra; ++a2)
                        sb += (long long)pick4r(d.ncls, a2) * K.mc *
                              ((pick4r(d.ncls, a2 ^ kc) + 3) & ~3);
                    off = K.off + sb + (long long)K.kpos * w;
                    stride = K.mc * w;
                } else {
                    n = N;
                    off = d.H_off + (long long)kl * N * d.Npad;
                    stride = d.Npad;
                }
            }
            for (int s = 0; s < NTM; ++s) {
                const int row = l0 + gl * s;
                for (int j = 0; j < L; j += 8) {
                    float v[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        v[e] = (row < ncl && j + e < n) ? P.H[off + (long long)row * stride + j + e]
                                                        : 0.f;
                    __syncwarp();
                    tmem_st8(taddr + (uint32_t)(j * NTM + 8 * s), v);
                }
            }
            tmem_wait_st();
            for (int s = 0; s < NSM; ++s) {
                const int row = l0 + gl * (NTM + s);
                for (int j = 0; j < L; ++j)
                    if (row < ncl && j < n)
                        reinterpret_cast<float *>(hsm + (s * (L / 4) + j / 4) * WT)[j & 3] =
                            P.H[off + (long long)row * stride + j];
            }
        }
        const float *const qcol = rhs + (cls ? (ra ^ kc) * QB : 0);
        const float *const qrow = rhs + ra * QB + l0;
        float *const fp = sm + O.fp + warp * R * 4 * QB + ra * QB + l0;

        // ---- update role: owned mode 32 chunk + lane.  The chunks go to the last
        // warps first (those without a stress mode, if any); the warps repeat them.
        const int wr = W - 1 - warp, reps = sub > 1 ? max(W / C, 1) : 1;
        const int chunk = wr % C, rep = wr / C;
        const int oi = 32 * chunk + lane;                       // owned index
        const bool upd = rep < reps;                            // this warp updates
        const bool on = upd && oi < no;
        const bool lead = on && rep == 0;                       // writes the mode's results
        // the warps that repeat a chunk share its sums and stores: bits 0..4 the
        // gradient sums, then w, q', v' of the segments and the pickup
        int duty = 0;
        for (int g = 0; g < 9; ++g)
            if (on && g % reps == rep) duty |= 1 << g;
        constexpr int kDutyW = 1 << 5, kDutyQ = 1 << 6, kDutyV = 1 << 7, kDutyY = 1 << 8;
        const long long m = d.mode_off + m0 + oi;
        float *const cf = sm + O.coef + tid;
        float *const ga = sm + O.gacc + tid;
        int cpos = 0;
        float y0 = 0.f, y1 = 0.f, y2 = 0.f, y3 = 0.f, x0 = 0.f, x1 = 0.f, x2 = 0.f;
        float qn1 = 0.f;
        if (on) {
            cpos = class_pos(m0 + oi);
            cf[0 * WT] = P.coef.eps[m];
            cf[1 * WT] = P.coef.rw2[m];
            cf[2 * WT] = P.coef.rw2lo[m];
            cf[3 * WT] = P.coef.r[m];
            cf[4 * WT] = P.coef.b[m];
            cf[5 * WT] = P.coef.c[m];
            cf[6 * WT] = P.coef.clo[m];
            if (FWD || FUSED) {
                y0 = rec0[m];
                y1 = rec0[TM + m];
                y2 = rec0[2 * TM + m];
                y3 = rec0[3 * TM + m];
            }
            if (REV) {
                x0 = P.adj[m];
                x1 = P.adj[TM + m];
                x2 = P.adj[2 * TM + m];
            }
        }
        // running addresses of the step's stored states
        const bool rec = FWD && P.mode == MODE_RECOMPUTE;
        float *pq = (FUSED ? P.rseg_q : P.seg_q) + m, *pv = (FUSED ? P.rseg_v : P.seg_v) + m;
        float *pw = P.seg_w ? P.seg_w + (long long)(rsteps - 1) * TM + m : nullptr;
        const float *pvn = REV ? P.seg_v + (long long)(rsteps - 2) * TM + m : nullptr;
        const bool st_q = (FUSED || rec) && (duty & kDutyQ), st_v = (FUSED || rec) && (duty & kDutyV);
        const bool st_w = REV && pw && (duty & kDutyW);
        auto store_state = [&]() {
            if (st_q) *pq = y0;
            if (st_v) *pv = y2;
            pq += TM;
            pv += TM;
        };
        auto store_ckpt = [&](int idx) {
            float *ck = P.ckpt + (long long)idx * kStateArrays * TM;
            ck[m] = y0;
            ck[TM + m] = y1;
            ck[2 * TM + m] = y2;
            ck[3 * TM + m] = y3;
        };
        const bool ckpt = FWD && P.mode == MODE_FORWARD && P.ckpt;
        int ck_left = P.ckpt_K, ck_idx = 1;                     // steps to the next checkpoint
        if (on) {
            if (ckpt && lead) store_ckpt(0);
            if (REV) {
                for (int g = 0; g < 2 * GA_N; ++g) ga[g * WT] = P.gacc[(long long)g * TM + m];
                qn1 = P.seg_q[(long long)rsteps * TM + m];
                sm[O.vst + tid] = P.seg_v[(long long)(rsteps - 1) * TM + m];
                if (st_w) *pw = cf[3 * WT] * x0;
            }
        }
        store_state();
        if (REV) pw -= TM;
        const float *const exc = P.exc ? P.exc + (long long)A.plate * P.total_steps : nullptr;
        const float *const yb = REV ? P.ybar + (long long)A.plate * P.total_steps : nullptr;
        // excitation and targets: a lane holds one of 32 steps
        float eb = 0.f, erb = 0.f, ybb = 0.f, ybn = 0.f;
        auto load_block = [&](int it) {
            const int i = it + lane, n = P.n_begin + (REV ? rsteps - 1 - i : i);
            eb = erb = ybb = 0.f;
            if (exc) {
                if (i < rsteps) eb = exc[n];
                if (FUSED && i < P.steps) erb = exc[P.rec_begin + i];
            }
            if (REV && i < rsteps && n >= 1) ybb = yb[n - 1];
        };
        if (REV) ybn = yb[P.n_begin + rsteps - 1];
        // q^n of the next step for every mode goes into the copy that is not read
        // (two modes per thread); this mode's v^n into its staging word
        const float *nq_src = REV ? P.seg_q + (long long)(rsteps - 2) * TM + d.mode_off + tid : nullptr;
        auto stage_next = [&](int it) {       // inputs of step it (< rsteps), into copy it & 1
            float *const nb = rhs + (it & 1) * 4 * QB;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (mon[h]) {
                    if (it < rsteps)
                        copy4(nb + mp[h], nq_src + h * WT);
                    else
                        nb[mp[h]] = 0.f;
                }
            nq_src -= TM;
        };
        if (REV) stage_next(1);
        float *px = (REV && P.xe && (d.has_dir || P.xe_all))
                        ? P.xe + (long long)(rsteps - 1) * 2 * P.total_k + d.k_off + kl : nullptr;
        const bool st_x = px && kon && lane == 0;
        const uint32_t tx_f = (uint32_t)(sub * no * XF * 4), tx_q = (uint32_t)(N * 4 * (FUSED ? 2 : 1));
        const uint32_t q_dst = su32(rhs + cpos + (REV ? bw : 0)), q_bar = su32(bar_q);
        const uint32_t q_dst0 = sub > 1 ? peer_addr(q_dst, (uint32_t)(A.base + min(rep, sub - 1))) : 0u;
        const uint32_t q_bar0 = sub > 1 ? peer_addr(q_bar, (uint32_t)(A.base + min(rep, sub - 1))) : 0u;
        const uint32_t y_dst0 = sub > 1 ? peer_addr(su32(sm + O.pick + 2 * (m0 + oi)), (uint32_t)(A.base + sub - 1)) : 0u;
        const uint32_t y_bar0 = sub > 1 ? peer_addr(su32(bar_y), (uint32_t)(A.base + sub - 1)) : 0u;
        const uint32_t xbuf = (uint32_t)(sub * Q.no_max * XF * 4);
        // the next phases are armed by a thread that has waited for the last ones
        const bool arms = sub > 1 && wr == 0 && lane == 0;
        bool dead = false;
        // a wait that runs out keeps the common control flow without further waits
        auto wait = [&](uint64_t *b, uint32_t parity) {
            if (dead) return;
            long long i = 0;
            while (!bar_try(b, parity) && ++i < kResWait) {
            }
            dead = i >= kResWait;
        };
        bar_sync_id(1, WT);

        for (int it = 0; it < P.steps; ++it) {
            const bool rev_on = REV && it < rsteps;
            const bool rev_next = REV && it + 1 < rsteps;
            const int buf = it & 1;
            const int qb = REV ? buf * 4 * QB : 0;
            if ((it & 31) == 0) load_block(it);
            // ---- row products, eta (xi, eta'), this warp's forces.  Rows and columns
            // beyond a class are zero, so nothing is guarded.
            float dot[R];
            if (kon) {
                const float *qs[R];
                qs[0] = qcol + qb;
                if constexpr (REV) qs[1] = qcol + bw;
                if constexpr (FUSED) qs[2] = qcol + br;
                float u[NR][R];
                row_products<R, NTM, NSM>(hsm, WT, taddr, L, qs, u);
#pragma unroll
                for (int x = 0; x < R; ++x) dot[x] = 0.f;
#pragma unroll
                for (int s = 0; s < NR; ++s) {
                    dot[0] = fmaf(qrow[qb + gl * s], u[s][0], dot[0]);
                    if constexpr (REV) dot[1] = fmaf(qrow[bw + gl * s], u[s][0], dot[1]);
                    if constexpr (FUSED) dot[2] = fmaf(qrow[br + gl * s], u[s][2], dot[2]);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int x = 0; x < R; ++x) dot[x] += __shfl_xor_sync(0xffffffffu, dot[x], o);
                const float ke = kap * dot[0];
#pragma unroll
                for (int s = 0; s < NR; ++s) {
                    if constexpr (FWD) {
                        fp[gl * s] = ke * u[s][0];
                    } else {
                        const float kx = kap * dot[1];
                        fp[gl * s] = fmaf(ke, u[s][1], 2.f * kx * u[s][0]);   // J w
                        fp[4 * QB + gl * s] = ke * u[s][0];                   // f(q^n)
                    }
                    if constexpr (FUSED) fp[8 * QB + gl * s] = (kap * dot[2]) * u[s][2];
                }
            }
            const float qn = REV ? rhs[qb + cpos] : 0.f;
            if (REV) copies_done();   // the next step's q^n (and this step's v^n) have arrived
            bar_sync_id(1, WT);       // the CTA's forces are in place, its right-hand sides read
            const int pb = (it / kPickSteps) & 1, ps = it % kPickSteps;
            if (pick_here && ps == 0 && it >= 2 * kPickSteps) bar_sync_id(4 + pb, WT + 32);
            // ---- forces of the CTA's stress modes (warps without one left zeros),
            // then of the plate
            auto cta_force = [&](int pos, float (&f)[R]) {
                const float *p = sm + O.fp + pos;
#pragma unroll
                for (int x = 0; x < R; ++x) f[x] = 0.f;
#pragma unroll
                for (int w = 0; w < kResMaxWarps; ++w)
#pragma unroll
                    for (int x = 0; x < R; ++x) f[x] += w < W ? p[(w * R + x) * 4 * QB] : 0.f;
            };
            float F[R];
#pragma unroll
            for (int x = 0; x < R; ++x) F[x] = 0.f;
            if (sub > 1) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (!mon[h]) continue;
                    float f[R];
                    cta_force(mp[h], f);
                    const uint32_t dst = mdst[h] + (buf ? xbuf : 0u);
                    if constexpr (R == 1) push1(dst, mbar[h], f[0]);
                    if constexpr (R == 2) push2(dst, mbar[h], f[0], f[1]);
                    if constexpr (R == 3) push4(dst, mbar[h], f[0], f[1], f[2]);
                }
                if (upd) {
                    wait(bar_f, (uint32_t)buf);
                    const float *x = sm + O.xch + (buf * sub * Q.no_max + oi) * XF;
                    if (on) {
#pragma unroll 8
                        for (int pr = 0; pr < sub; ++pr, x += Q.no_max * XF) {
                            if constexpr (R == 1) {
                                F[0] += x[0];
                            } else if constexpr (R == 2) {
                                const float2 v = *reinterpret_cast<const float2 *>(x);
                                F[0] += v.x;
                                F[1] += v.y;
                            } else {
                                const float4 v = *reinterpret_cast<const float4 *>(x);
                                F[0] += v.x;
                                F[1] += v.y;
                                F[2] += v.z;
                            }
                        }
                    }
                }
            } else if (on) {
                cta_force(cpos, F);
            }
            // ---- update and the new right-hand sides
            const float a_old = x0;
            float rr = 0.f, bcf = 0.f, cw = 0.f, wv = 0.f;
            const float e = __shfl_sync(0xffffffffu, eb, it & 31);
            const float er = FUSED ? __shfl_sync(0xffffffffu, erb, it & 31) : 0.f;
            const float ybm = REV ? __shfl_sync(0xffffffffu, ybb, it & 31) : 0.f;
            if (upd) {
                rr = cf[3 * WT];
                bcf = cf[4 * WT];
                cw = cf[5 * WT];
                if (REV && rev_on) adj_step(x0, x1, x2, cf[0 * WT], cf[1 * WT], F[0], cw * ybm);
                if (rev_next) wv = rr * x0;
                if (FWD || FUSED)
                    sv_step(y0, y1, y2, y3, cf[0 * WT], cf[1 * WT], cf[2 * WT], rr,
                            fmaf(bcf, FWD ? e : er, -F[FUSED ? 2 : 0]));
                if (sub > 1) {
                    if (on && rep < sub) {
                        push1(q_dst0, q_bar0, REV ? wv : y0);
                        if (FUSED) push1(q_dst0 + (uint32_t)((br - bw) * 4), q_bar0, y0);
                        for (int pr = rep + reps; pr < sub; pr += reps) {
                            const uint32_t qa = peer_addr(q_dst, (uint32_t)(A.base + pr));
                            const uint32_t ba = peer_addr(q_bar, (uint32_t)(A.base + pr));
                            push1(qa, ba, REV ? wv : y0);
                            if (FUSED) push1(qa + (uint32_t)((br - bw) * 4), ba, y0);
                        }
                    }
                } else {
                    if (on) {
                        if (FWD) rhs[cpos] = y0;
                        if (REV) rhs[bw + cpos] = wv;
                        if (FUSED) rhs[br + cpos] = y0;
                    }
                    __syncwarp();
                    if (lane == 0) bar_arrive(bar_q);
                }
            }
            // ---- off the chain: gradient sums, stores, pickups, the next step's inputs
            if (arms && it + 1 < P.steps) bar_expect_tx(bar_f, tx_f);
            if (REV && rev_on && kon) {
                kahan_add(ks, kcmp, -dot[0] * dot[1]);
                if (st_x) {
                    px[0] = dot[1];
                    px[P.total_k] = dot[0];
                }
            }
            if (REV) px -= 2 * P.total_k;
            if (REV && on && rev_on) {
                auto acc = [&](int idx, float x) {
                    if (!(duty & (1 << idx))) return;
                    float gs = ga[(2 * idx) * WT], gc = ga[(2 * idx + 1) * WT];
                    kahan_add(gs, gc, x);
                    ga[(2 * idx) * WT] = gs;
                    ga[(2 * idx + 1) * WT] = gc;
                };
                acc(GA_A, a_old * qn);
                acc(GA_V, a_old * sm[O.vst + tid]);
                acc(GA_F, a_old * fmaf(bcf, e, -F[R > 1 ? 1 : 0]));
                acc(GA_E, a_old * e);
                acc(GA_C, ybn * qn1);
                qn1 = qn;
                if (rev_next) {
                    if (st_w) *pw = wv;
                    if (duty & (1 << GA_V)) copy4(sm + O.vst + tid, pvn);
                }
            }
            if (REV) {
                pw -= TM;
                pvn -= TM;
                ybn = ybm;
                stage_next(it + 2);
            }
            if (FUSED || rec) store_state();
            if (on) {
                if (ckpt && ck_left == 1 && it + 1 < P.steps && lead) store_ckpt(ck_idx);
                if (FWD && (duty & kDutyY)) {
                    // pickup terms of eight steps, summed by the last rank's spare warp
                    float ys = 0.f, ye = 0.f;
                    pickup_add(ys, ye, cw, cf[6 * WT], y0, y1);
                    const int po = (pb * kPickSteps + ps) * O.PS;
                    if (sub > 1)
                        push2(y_dst0 + (uint32_t)(po * 4), y_bar0 + 8u * pb, ys, ye);
                    else
                        *reinterpret_cast<float2 *>(sm + O.pick + po + 2 * (m0 + oi)) =
                            make_float2(ys, ye);
                }
            }
            if (ckpt && --ck_left == 0) {
                ck_left = P.ckpt_K;
                ++ck_idx;
            }
            if (FWD && sub == 1 && (ps == kPickSteps - 1 || it == P.steps - 1))
                bar_arrive_id(2 + pb, WT + 32);
            wait(bar_q, (uint32_t)buf);
            if (arms && it + 1 < P.steps) bar_expect_tx(bar_q, tx_q);
        }

        // ---- write back
        if (lead) {
            if (FWD && P.mode == MODE_FORWARD) {
                P.state_io[m] = y0;
                P.state_io[TM + m] = y1;
                P.state_io[2 * TM + m] = y2;
                P.state_io[3 * TM + m] = y3;
            }
            if (REV) {
                P.adj[m] = x0;
                P.adj[TM + m] = x1;
                P.adj[2 * TM + m] = x2;
            }
        }
        if (REV && on)
            for (int g = 0; g < GA_N; ++g)
                if (duty & (1 << g)) {
                    P.gacc[(long long)(2 * g) * TM + m] = ga[(2 * g) * WT];
                    P.gacc[(long long)(2 * g + 1) * TM + m] = ga[(2 * g + 1) * WT];
                }
        if (REV && kon && lane == 0) {
            P.kacc[2 * (d.k_off + kl)] = ks;
            P.kacc[2 * (d.k_off + kl) + 1] = kcmp;
        }
        if (dead && lane == 0) set_status(P.status, A.plate, MDX_ERR_TIMEOUT);
    } else if (pick_here && warp == W) {
        // ======================================================== spare warp: pickups
        // lane = 4 ps + part: a quarter of the modes of one of eight steps
        const int ps = lane >> 2, part = lane & 3;
        bool bad = false, dead = false;
        for (int i0 = 0; i0 < P.steps; i0 += kPickSteps) {
            const int grp = i0 / kPickSteps, pb = grp & 1;
            const int cnt = min(kPickSteps, P.steps - i0);
            if (sub > 1) {
                if (lane == 0) bar_expect_tx(bar_y + pb, (uint32_t)(cnt * N * 8));
                long long i = 0;
                while (!dead && !bar_try(bar_y + pb, (uint32_t)((grp >> 1) & 1)) &&
                       ++i < 16 * kResWait) {
                }
                if (i >= 16 * kResWait) dead = true;
                __syncwarp();
            } else {
                bar_sync_id(2 + pb, WT + 32);
            }
            const float *pk = sm + O.pick + (pb * kPickSteps + ps) * O.PS;
            float ys = 0.f, ye = 0.f;
            if (ps < cnt)
                for (int j = part; j < N; j += 4) {
                    const float2 v = *reinterpret_cast<const float2 *>(pk + 2 * j);
                    pickup_merge(ys, ye, v.x, v.y);
                }
#pragma unroll
            for (int o = 1; o <= 2; o <<= 1) {
                const float s2 = __shfl_xor_sync(0xffffffffu, ys, o);
                const float e2 = __shfl_xor_sync(0xffffffffu, ye, o);
                pickup_merge(ys, ye, s2, e2);
            }
            // the buffer is free for the steps two groups on
            if (i0 + 2 * kPickSteps < P.steps) bar_arrive_id(4 + pb, WT + 32);
            const float y = ys + ye;
            if (part == 0 && ps < cnt) {
                if (P.mode == MODE_FORWARD && P.audio)
                    P.audio[(long long)A.plate * P.total_steps + P.n_begin + i0 + ps] = y;
                if (!isfinite(y)) bad = true;
            }
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) set_status(P.status, A.plate, MDX_ERR_NONFINITE);
        if (dead && lane == 0) set_status(P.status, A.plate, MDX_ERR_TIMEOUT);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem0), "r"(Q.tcols)
                     : "memory");
    // no CTA leaves while a peer may still store into its shared memory
    cluster_sync_all();
}

namespace {

// Kernel variants by longest row: a lane's rows in tensor memory (256 words a
// thread with more than four warps, else 512) and the rest in shared memory.
constexpr int kVarLen[kResVariants] = {16, 24, 32, 40, 48, 56, 64};
constexpr int kVarTm[kResVariants] = {2, 2, 4, 4, 4, 4, 6};
constexpr int kVarSm[kResVariants] = {0, 1, 0, 1, 2, 3, 2};
// the spare warp makes eight: 255 registers a thread
int var_warps(int v) { return kVarTm[v] * kVarLen[v] > 256 ? 4 : kResMaxWarps; }

template <int R>
const void *res_fn_r(int v) {
    switch (v) {
        case 0: return reinterpret_cast<const void *>(resident_kernel<R, 2, 0, 16>);
        case 1: return reinterpret_cast<const void *>(resident_kernel<R, 2, 1, 24>);
        case 2: return reinterpret_cast<const void *>(resident_kernel<R, 4, 0, 32>);
        case 3: return reinterpret_cast<const void *>(resident_kernel<R, 4, 1, 40>);
        case 4: return reinterpret_cast<const void *>(resident_kernel<R, 4, 2, 48>);
        case 5: return reinterpret_cast<const void *>(resident_kernel<R, 4, 3, 56>);
        default: return reinterpret_cast<const void *>(resident_kernel<R, 6, 2, 64>);
    }
}

const void *res_fn(int r, int v) {
    return r == 1 ? res_fn_r<1>(v) : (r == 2 ? res_fn_r<2>(v) : res_fn_r<3>(v));
}

void res_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *at, int grid, int cs, int threads,
                size_t smem, cudaStream_t s) {
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
}

}  // namespace

// Variant for rows of w columns held by `rows` rows a lane (-1: none), and the
// most warps (stress modes) of its CTAs.
int resident_variant(int w, int rows) {
    for (int v = 0; v < kResVariants; ++v)
        if (w <= kVarLen[v] && rows <= kVarSm[v] + kVarTm[v]) return v;
    return -1;
}
int resident_max_warps(int variant) { return var_warps(variant); }

// Tensor-memory columns of a launch: the thread-private words of its rows,
// twice where eight warps share the four lane quarters.
int resident_columns(int variant, int L, int warps) {
    const int words = kVarTm[variant] * L * (warps > 4 ? 2 : 1);
    int c = 32;
    while (c < words) c *= 2;
    return c;
}

// Dynamic shared memory of a launch.  The request is at least the share of the
// SM's shared memory that the launch takes of its tensor memory, so CTAs that
// fit an SM together (of this or another launch) never wait for each other's
// columns: a CTA whose cluster peers wait must not block on an allocation.
size_t resident_smem(int R, const ResidentParams &Q) {
    const ResLayout o = res_layout(R, Q.warps, kVarLen[Q.variant], Q.L, Q.n_max, Q.no_max,
                                    Q.max_sub, kVarSm[Q.variant]);
    return std::max(sizeof(float) * (size_t)o.end, (size_t)Q.tcols * kSmemPerColumn);
}

// Sets the kernels' attributes and returns how many clusters of cs CTAs run at
// once (0: the shape cannot be launched).
cudaError_t resident_check(int cs, const ResidentParams &Q, size_t smem_optin, int *fit) {
    *fit = 1 << 30;
    for (int r = 1; r <= 3; ++r) {
        const void *fn = res_fn(r, Q.variant);
        const size_t smem = resident_smem(r, Q);
        if (smem + kResStatic > smem_optin) {
            *fit = 0;
            return cudaSuccess;
        }
        // attributes belong to the kernels, not to a plan: only ever raised
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(smem_optin - kResStatic));
        if (e == cudaSuccess && cs > 8)
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at[1];
        res_config(cfg, at, cs, cs, 32 * Q.warps + (r == 1 ? 32 : 0), smem, nullptr);
        int n = 0;
        e = cudaOccupancyMaxActiveClusters(&n, fn, &cfg);
        if (e != cudaSuccess) return e;
        *fit = std::min(*fit, n);
    }
    return cudaSuccess;
}

cudaError_t launch_resident(int R, const ResidentParams &Q, int grid, int cs, size_t smem,
                            cudaStream_t s) {
    if (grid <= 0 || Q.p.steps <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    res_config(cfg, at, grid, cs, 32 * Q.warps + (R == 1 ? 32 : 0), smem, s);
    ResidentParams q = Q;
    void *args[] = {&q};
    return cudaLaunchKernelExC(&cfg, res_fn(R, Q.variant), args);
}

}  // namespace mdx
