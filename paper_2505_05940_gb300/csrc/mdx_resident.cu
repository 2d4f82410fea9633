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
// clusters that do not fit at once run one after the other.  Measured, streaming
// and here: 100 x 30 plate, 11 025 steps, 34.3 and 13.1 ms; 96 plates of 50 to
// 200 modes 196 and 37.5 ms; a fit's step (forward with checkpoints, recompute and
// reverse) of 6 plates of 117 x 29, 3 001 steps, 79.6 and 14.0 ms, of 64 plates of
// 200 x 50, 4 410 steps, 346 and 219 ms.
//
// Rows: one warp per stress mode k.  Lanes 8 a .. 8 a + 7 hold the rows of
// class a (row l + 8 r of the class in lane l, register row r), whose only
// nonzero columns are those of class a ^ class(k), so all rows of a lane share
// their right-hand-side loads (four broadcast addresses a warp, one wavefront)
// and eta_k is a sum within the warp: no barrier before the forces.  A plate
// without classes (N <= 64) spreads its rows over the 32 lanes.  The rows live
// in tensor memory (NTM rows), used as a thread-private extension of the
// register file, the others in registers (NREG, checkpoint-free passes) or shared
// memory (NSM).  Tensor memory rather than shared memory: reading 224 words a
// thread with their FMAs took 512 cycles per CTA of 256 threads (448 of them the
// FMAs), from shared memory (LDS.128) 1 800.  Products are packed FMAs (two
// columns at a time).
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
// Order of the sums: a gradient's last digits follow the forward states', so
// the passes with checkpoints keep the streaming kernel's order of every sum
// (ORD 1, 2).  Products alternate between two chains per row (the halves of the
// packed FMAs); the streaming kernel starts them anew with each stage of rows, so
// behind a stage of an odd number of rows they change sides, here a zero column
// (and a layout of the right-hand sides with that gap).  The force adds one chain
// per run of stress modes; a CTA stores the runs that end in it as separate parts
// and hands the one that goes on to the next CTA.
//
// Pickups: one warp per chunk of owned modes keeps its terms and sums them every
// eight steps (with shuffles every step this was 320 cycles of the step's chain);
// one warp of the last rank adds the chunks' terms.
//
// Bound: the dependent chain of a step (one barrier, one warp reduction, two
// exchanges of 400 cycles, the update; some 770 instructions a warp at 5 cycles)
// plus the packed FMAs: 100 x 30 modes on 8 CTAs take 2 490 cycles a step, 620 of
// them products; 196 x 49 on 7 CTAs 3 860 and 1 740; the fused sweep of 200 x 50
// on 10 CTAs 11 300 and 4 950.
#include <cuda_runtime.h>

#include <algorithm>

#include "../../include/mdx.h"
#include "mdx_common.cuh"
#include "mdx_tc.cuh"

namespace mdx {

namespace {

using namespace tc;

typedef unsigned long long u64;

constexpr int kResMaxWarps = 8;              // warps of a CTA
constexpr int kPickSteps = 8;                // pickups reduced together
constexpr int kPickPitch = 36;               // terms of a step: 4 lanes x 4 steps on distinct banks

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
// host.  W warps, kernel row length LM, NO owned modes and segs parts at most.
struct ResLayout {
    int QB, PS;                 // class block, pickup terms per step
    int LF;                     // right-hand sides of one layout
    int rhs, fp, ke, xch, car, lp, dp, hs, coef, pick, pst, gacc, vst, end;
};

__host__ __device__ inline ResLayout res_layout(int R, int LM, const ResidentParams &Q, int nsm) {
    const int W = Q.warps, L = Q.L, NO = Q.no_max, sub = Q.max_sub, segs = Q.segs;
    ResLayout o;
    // class blocks 8 banks apart, so that the four classes' accesses do not collide
    o.QB = ((LM + 31) & ~31) + 8;
    o.PS = sub * ((NO + 31) / 32);
    int p = 16;                 // mbarriers, tensor-memory base
    o.LF = rhs_blocks(R) * 4 * o.QB;
    o.rhs = p;                  // [layouts][blocks][4][QB]
    p += Q.lays * o.LF + 8;     // (a chunk is read past the last block)
    o.fp = p;                   // [W][R][4][QB] products of each warp's stress mode
    p += W * R * 4 * o.QB;
    o.ke = p;                   // [W][8] its factors of the forces
    p += W * 8;
    o.xch = p;                  // [2][segs][NO] x (1, 2 or 4 floats): parts of the owned modes
    if (sub > 1) p += 2 * segs * NO * (R == 3 ? 4 : R);
    p = (p + 3) & ~3;
    o.car = p;                  // [2][n_max] x (1, 2 or 4 floats): parts begun in the CTA before
    if (Q.carry) p += 2 * Q.n_max * (R == 3 ? 4 : R);
    o.lp = p;                   // [layouts - 1][64 W] places of the plate's modes (ints)
    p += (Q.lays - 1) * 64 * W;
    o.dp = p;                   // [sub][layouts][NO] places of the owned modes in a peer's layouts,
    if (Q.lays > 1) p += sub * Q.lays * NO;   // row 0: their number
    p = (p + 3) & ~3;
    o.hs = p;                   // [nsm][L / 4][32 W] x 4: coupling rows (thread-private)
    p += nsm * L * 32 * W;
    o.coef = p;                 // [7][32 W] coefficients of the updated modes
    p += 7 * 32 * W;
    p = (p + 1) & ~1;
    o.pick = p;                 // [2][kPickSteps][PS] x 2: pickup terms of the owners' chunks
    if (R == 1) p += 2 * kPickSteps * 2 * o.PS;
    o.pst = p;                  // [chunks][kPickSteps][kPickPitch] x 2: a chunk's terms of its modes
    if (R == 1) p += (NO + 31) / 32 * kPickSteps * kPickPitch * 2;
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
// One warp's products u[r][x] = sum_j H[r][j] q_x[j] over NTM tensor-memory
// rows ([column / 8][row][8], read two rows at a time, the next pair in flight
// during this pair's FMAs), NSM shared-memory rows and NREG register rows.  A
// chunk's shared-memory rows are loaded before and multiplied after its
// tensor-memory rows, so the two warps of a scheduler do not alternate between
// loading and multiplying.  Without register rows the loop over the columns
// stays rolled.  SP chains per row (two where few rows leave the FMAs' latency
// uncovered).
template <int R, int NTM, int NSM, int NREG, int LMAX, int SP>
__device__ __forceinline__ void row_products(const float4 *hs, int hs_stride, uint32_t taddr, int L,
                                             const u64 (&hr)[NREG > 0 ? NREG : 1][LMAX / 2],
                                             const float *const (&q)[R], float (&u)[NTM + NSM + NREG][R]) {
    constexpr int NA = NTM + NSM + NREG, NP = NTM / 2;
    // all rows in tensor memory: the next right-hand sides are loaded during the
    // FMAs (1.40 instead of 1.44 us a step at 100 x 30); not worth its registers
    // where other rows' loads cover theirs (4.15 / 3.93 us at 96 plates)
    constexpr bool PF = NA == NTM;
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
    ulonglong2 qv[2][R][2];
    auto load_q = [&](int j, ulonglong2 (&d)[R][2]) {
#pragma unroll
        for (int x = 0; x < R; ++x) {
            d[x][0] = *reinterpret_cast<const ulonglong2 *>(q[x] + j);
            d[x][1] = *reinterpret_cast<const ulonglong2 *>(q[x] + j + 4);
        }
    };
    auto mac = [&](u64 (&a)[SP], u64 h0, u64 h1, u64 h2, u64 h3, const ulonglong2 (&v)[2]) {
        a[0] = ffma2(h0, v[0].x, a[0]);
        a[SP - 1] = ffma2(h1, v[0].y, a[SP - 1]);
        a[0] = ffma2(h2, v[1].x, a[0]);
        a[SP - 1] = ffma2(h3, v[1].y, a[SP - 1]);
    };
    // columns j .. j + 7; h: parity of j / 8
    auto chunk = [&](int j, int h) {
        const float4 *hp = hs + (j / 4) * hs_stride;
        ulonglong2 ha[NSM > 0 ? NSM : 1], hb[NSM > 0 ? NSM : 1];
        if constexpr (!PF) load_q(j, qv[h]);
#pragma unroll
        for (int s = 0; s < NSM; ++s) {
            ha[s] = *reinterpret_cast<const ulonglong2 *>(hp + s * row4);
            hb[s] = *reinterpret_cast<const ulonglong2 *>(hp + s * row4 + hs_stride);
        }
        // (beyond the last chunk the padding of the block is read)
        if constexpr (PF) load_q(j + 8, qv[h ^ 1]);
#pragma unroll
        for (int g = 0; g < NP; ++g) {
            const int par = (h * NP + g) & 1;
            uint32_t (&w)[16] = tm[par];
            tmem_wait_ld(w);
            // beyond the last chunk the first pair is read again and not used
            const bool more = g + 1 < NP || j + 8 < L;
            tmem_ld_rows2(taddr + (uint32_t)(more ? j * NTM + 16 * (g + 1) : 0), tm[par ^ 1]);
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int x = 0; x < R; ++x)
                    mac(acc[2 * g + s][x], pack2(w[8 * s], w[8 * s + 1]), pack2(w[8 * s + 2], w[8 * s + 3]),
                        pack2(w[8 * s + 4], w[8 * s + 5]), pack2(w[8 * s + 6], w[8 * s + 7]), qv[h][x]);
        }
#pragma unroll
        for (int s = 0; s < NSM; ++s)
#pragma unroll
            for (int x = 0; x < R; ++x)
                mac(acc[NTM + s][x], ha[s].x, ha[s].y, hb[s].x, hb[s].y, qv[h][x]);
    };
    if constexpr (PF) load_q(0, qv[0]);
    if constexpr (NREG > 0) {
#pragma unroll
        for (int j = 0; j < LMAX; j += 8) {
            if (j >= L) break;
            chunk(j, (j / 8) & 1);
#pragma unroll
            for (int s = 0; s < NREG; ++s)
#pragma unroll
                for (int x = 0; x < R; ++x)
                    mac(acc[NTM + NSM + s][x], hr[s][j / 2], hr[s][j / 2 + 1], hr[s][j / 2 + 2], hr[s][j / 2 + 3],
                        qv[(j / 8) & 1][x]);
        }
    } else {
#pragma unroll 1
        for (int j = 0; j < L; j += 16) {
            chunk(j, 0);
            if (j + 8 >= L) break;
            chunk(j + 8, 1);
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

// The one row a lane holds of a plate without classes (N <= 32): rounded products
// added in column order, as the streaming kernel's row groups combine them.
template <int R, int NTM>
__device__ __forceinline__ void dense_row(uint32_t taddr, int L, const float *const (&q)[R], float (&u)[R]) {
#pragma unroll
    for (int x = 0; x < R; ++x) u[x] = 0.f;
#pragma unroll 1
    for (int j = 0; j < L; j += 8) {
        uint32_t w[16];
        tmem_ld_rows2(taddr + (uint32_t)(j * NTM), w);
        tmem_wait_ld(w);
#pragma unroll
        for (int e = 0; e < 8; ++e)
#pragma unroll
            for (int x = 0; x < R; ++x)
                u[x] = __fadd_rn(u[x], __fmul_rn(__uint_as_float(w[e]), q[x][j + e]));
    }
}

}  // namespace

// ORD: the order of the sums.  0: the fastest; 1, 2: the streaming kernel's, digit
// for digit, 2 also where rows have gaps or a part spans CTAs (kept out of the
// others: its code alone cost them 3 to 11 % of a step).
template <int R, int NTM, int NSM, int NREG, int LMAX, int ORD>
__global__ void __launch_bounds__(256, 1) resident_kernel(const ResidentParams Q) {
    extern __shared__ __align__(16) float sm[];
    __shared__ ResCta A;
    __shared__ InstDesc d;
    __shared__ int gave_up;                       // a wait of this CTA ran out
    const PlateParams &P = Q.p;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr bool REV = R >= 2, FWD = R == 1, FUSED = R == 3;
    constexpr bool SAME = ORD > 0, EXT = ORD == 2;
    constexpr int NR = NTM + NSM + NREG;          // rows of a lane
    constexpr int XF = R == 3 ? 4 : R;            // floats per exchanged entry
    constexpr int QB = ((LMAX + 31) & ~31) + 8;
    const int W = Q.warps, WT = 32 * W;
    const ResLayout O = res_layout(R, LMAX, Q, NSM);
    uint64_t *bar_f = reinterpret_cast<uint64_t *>(sm);        // forces of the owned modes
    uint64_t *bar_q = bar_f + 1;                               // new right-hand sides
    uint64_t *bar_y = bar_f + 2;                               // pickup terms (two buffers)
    uint32_t *tbase = reinterpret_cast<uint32_t *>(sm + 8);
    uint64_t *bar_c = reinterpret_cast<uint64_t *>(sm + 10);   // parts begun in the CTA before
    const long long TM = P.total_modes;
    for (int e = tid; e < (int)(sizeof(ResCta) / 4); e += blockDim.x)
        reinterpret_cast<int *>(&A)[e] = reinterpret_cast<const int *>(Q.ctas + blockIdx.x)[e];
    for (int e = 16 + tid; e < O.end; e += blockDim.x) sm[e] = 0.f;
    if (tid == 0) gave_up = 0;
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
    const int lays = EXT && used ? A.lays : 1;
    const bool more_lays = EXT && Q.lays > 1;
    if (tid == 0) {
        bar_init(bar_f, 1);
        bar_init(bar_q, sub > 1 ? 1 : C);
        bar_init(bar_y, 1);
        bar_init(bar_y + 1, 1);
        bar_init(bar_c, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (sub > 1) {
            if (no > 0) bar_expect_tx(bar_f, (uint32_t)(A.segs_all * no * XF * 4));
            bar_expect_tx(bar_q, (uint32_t)(N * 4 * (FUSED ? 2 : 1) * lays));
            if (EXT && (A.carry & 1)) bar_expect_tx(bar_c, (uint32_t)(N * XF * 4));
        }
    }
    // class row of a user-order mode, and its place in a right-hand-side block
    auto class_pos = [&](int i) {
        if (!cls) return i;
        const int row = Q.iperm[d.perm_off + i];
        const int a = (row >= d.ocls[1]) + (row >= d.ocls[2]) + (row >= d.ocls[3]);
        return a * QB + row - pick4r(d.ocls, a);
    };
    // the same in layout l of a CTA
    auto lay_pos = [&](const ResCta &c, int l, int pos) {
        const int a = pos / QB, i = pos - a * QB, g = c.gap[l - 1][a];
        return l * O.LF + pos + (g > 0 ? i / g : 0);
    };
    float *const rhs = sm + O.rhs;
    int *const lp = reinterpret_cast<int *>(sm + O.lp) + tid, *const dp = reinterpret_cast<int *>(sm + O.dp);
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
    if (used) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = tid + h * WT;
            if (i >= N) continue;
            // (bit 5 of the debug flags: the second CTA of a plate withholds its parts)
            mon[h] = !((P.debug_flags & 32) && rank == 1);
            const long long m = d.mode_off + i;
            mp[h] = class_pos(i);
            if (sub > 1) {
                const int own = ((i + 1) * sub - 1) / N;
                const int o0 = (int)((long long)N * own / sub);
                mdst[h] = peer_addr(su32(sm + O.xch) + (uint32_t)((A.seg0 * Q.no_max + i - o0) * XF * 4),
                                    (uint32_t)(A.base + own));
                mbar[h] = peer_addr(su32(bar_f), (uint32_t)(A.base + own));
            }
            for (int l = 0; l < lays; ++l) {
                const int at = l == 0 ? mp[h] : lay_pos(A, l, mp[h]);
                if (l > 0) lp[((l - 1) * 2 + h) * WT] = at;
                if (FWD) rhs[at] = rec0[m];
                if (REV) {
                    rhs[at] = P.seg_q[(long long)(rsteps - 1) * TM + m];
                    rhs[bw + at] = P.coef.r[m] * P.adj[m];
                }
                if (FUSED) rhs[br + at] = rec0[m];
            }
        }
    }
    // the owned modes' places in every CTA of the plate
    if (more_lays && used)
        for (int e = tid; e < sub * no; e += WT) {
            const int pr = e / no, oi = e - pr * no;
            const ResCta &c = Q.ctas[(int)blockIdx.x - rank + pr];
            const int pos = class_pos(m0 + oi);
            int *const row = dp + pr * Q.lays * Q.no_max + oi;
            row[0] = c.lays;
            for (int l = 1; l < c.lays; ++l) row[l * Q.no_max] = lay_pos(c, l, pos) - pos;
        }
    __syncthreads();
    cluster_sync_all();      // every peer's barriers exist before the first store

    if (used) {
        // ---- row role: rows of stress mode k0 + warp
        const bool kon = warp < nk;
        const int ra = cls ? lane >> 3 : 0;
        const int gl = cls ? 8 : 32, l0 = cls ? lane & 7 : lane;
        const int kl = A.k0 + warp;
        int kc = 0;
        const uint32_t taddr = tmem0 + ((uint32_t)(32 * (warp & 3)) << 16) +
                               (warp >= 4 ? (uint32_t)(Q.tcols / 2) : 0u);
        float4 *const hsm = reinterpret_cast<float4 *>(sm + O.hs) + tid;
        u64 hreg[NREG > 0 ? NREG : 1][LMAX / 2];                // register rows
        float kap = 0.f, ks = 0.f, kcmp = 0.f;                  // kappa, d kappa (Kahan)
        {
            const int ncl = cls ? pick4r(d.ncls, ra) : N;       // rows of this lane's class
            // element (row, j) at off + j stride + row: a row of H^k is read as the
            // column the streaming kernel sums (H need not be symmetric to the last bit)
            long long off = 0;
            int n = 0, stride = 0;
            const int lay = EXT && kon ? A.lay_of >> (4 * warp) & 15 : 0;
            int gap = 0;                                        // a zero column after every gap
            if (kon) {
                kap = P.kappa[d.k_off + kl];
                if (REV) {
                    ks = P.kacc[2 * (d.k_off + kl)];
                    kcmp = P.kacc[2 * (d.k_off + kl) + 1];
                }
                if (cls) {
                    const ClusterK K = Q.kinfo[d.k_off + kl];
                    kc = K.c;
                    const int w = (ncl + 3) & ~3;
                    n = pick4r(d.ncls, ra ^ kc);
                    if (lay > 0) gap = A.gap[lay - 1][ra ^ kc];
                    long long sb = 0;
                    for (int a2 = 0; a2 < (ra ^ kc); ++a2)
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
            auto element = [&](int row, int p) {
                const int s = gap > 0 ? p / (gap + 1) : 0, j = p - s;
                const bool in = row < ncl && j < n && (gap == 0 || p - s * (gap + 1) < gap);
                return in ? P.H[off + (long long)j * stride + row] : 0.f;
            };
            for (int s = 0; s < NTM; ++s) {
                const int row = l0 + gl * s;
                for (int j = 0; j < L; j += 8) {
                    float v[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[e] = element(row, j + e);
                    __syncwarp();
                    tmem_st8(taddr + (uint32_t)(j * NTM + 8 * s), v);
                }
            }
            tmem_wait_st();
            for (int s = 0; s < NSM; ++s) {
                const int row = l0 + gl * (NTM + s);
                for (int j = 0; j < L; ++j)
                    reinterpret_cast<float *>(hsm + (s * (L / 4) + j / 4) * WT)[j & 3] = element(row, j);
            }
#pragma unroll
            for (int s = 0; s < NREG; ++s) {
                const int row = l0 + gl * (NTM + NSM + s);
#pragma unroll
                for (int j = 0; j < LMAX; j += 2) {
                    float v[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) v[e] = element(row, j + e);
                    hreg[s][j / 2] = pack2(__float_as_uint(v[0]), __float_as_uint(v[1]));
                }
            }
        }
        const float *const qcol = rhs + (cls ? (ra ^ kc) * QB : 0) +
                                  (EXT && kon ? (int)(A.lay_of >> (4 * warp) & 15) * O.LF : 0);
        const float *const qrow = rhs + ra * QB + l0;
        float *const fpw = sm + O.fp + warp * R * 4 * QB, *const fp = fpw + ra * QB + l0;
        float *const kew = sm + O.ke;

        // ---- update role: owned mode 32 chunk + lane.  The chunks go to the last
        // warps first (those without a stress mode, if any); the warps repeat them.
        const int wr = W - 1 - warp, reps = sub > 1 ? max(W / C, 1) : 1;
        const int chunk = wr % C, rep = wr / C;
        const int oi = 32 * chunk + lane;                       // owned index
        // This warp updates.  None does in a CTA without modes (more CTAs than modes): it
        // receives no parts, and a phase of bar_f without bytes ends by being armed, so
        // it would run ahead of a warp that waited for it.
        const bool upd = rep < reps && no > 0;
        bool on = upd && oi < no;
        const bool lead = on && rep == 0;                       // writes the mode's results
        // the warps that repeat a chunk share its sums and stores: bits 0..4 the
        // gradient sums, then w, q', v' of the segments
        int duty = 0;
        for (int g = 0; g < 8; ++g)
            if (on && g % reps == rep) duty |= 1 << g;
        constexpr int kDutyW = 1 << 5, kDutyQ = 1 << 6, kDutyV = 1 << 7;
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
        const bool rec = SAME && FWD && P.mode == MODE_RECOMPUTE;
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
        const bool ckpt = SAME && FWD && P.mode == MODE_FORWARD && P.ckpt;
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
                    if (more_lays)
#pragma unroll 1
                        for (int l = 0; l < lays - 1; ++l) {
                            const int at = lp[(l * 2 + h) * WT];
                            if (it < rsteps)
                                copy4(nb + at, nq_src + h * WT);
                            else
                                nb[at] = 0.f;
                        }
                }
            nq_src -= TM;
        };
        if (REV) stage_next(1);
        float *px = (REV && P.xe && (d.has_dir || P.xe_all))
                        ? P.xe + (long long)(rsteps - 1) * 2 * P.total_k + d.k_off + kl : nullptr;
        const bool st_x = px && kon && lane == 0;
        const uint32_t tx_f = (uint32_t)(A.segs_all * no * XF * 4), tx_q = (uint32_t)(N * 4 * (FUSED ? 2 : 1) * lays);
        const uint32_t q_dst = su32(rhs + cpos + (REV ? bw : 0)), q_bar = su32(bar_q);
        const uint32_t q_dst0 = sub > 1 ? peer_addr(q_dst, (uint32_t)(A.base + min(rep, sub - 1))) : 0u;
        const uint32_t q_bar0 = sub > 1 ? peer_addr(q_bar, (uint32_t)(A.base + min(rep, sub - 1))) : 0u;
        // pickups: a warp per chunk sums its modes' terms every step; one warp of the
        // last rank adds the chunks' terms, eight steps at a time
        const bool picks = FWD && upd && rep == 0;
        const bool collects = FWD && upd && rank == sub - 1 && wr == 0;
        const int cmax = ((N + sub - 1) / sub + 31) / 32, yent = rank * cmax + chunk;
        int chunks_all = 0;
        for (int r = 0; r < sub; ++r)
            chunks_all += ((int)((long long)N * (r + 1) / sub) - (int)((long long)N * r / sub) + 31) / 32;
        float2 *const pst = reinterpret_cast<float2 *>(sm + O.pst) + chunk * kPickSteps * kPickPitch;
        const uint32_t y_dst0 = sub > 1 ? peer_addr(su32(sm + O.pick + 2 * yent), (uint32_t)(A.base + sub - 1)) : 0u;
        const uint32_t y_bar0 = sub > 1 ? peer_addr(su32(bar_y), (uint32_t)(A.base + sub - 1)) : 0u;
        auto arm_y = [&](int grp) {
            const int cnt = min(kPickSteps, P.steps - grp * kPickSteps);
            if (sub > 1 && cnt > 0 && lane == 0) bar_expect_tx(bar_y + (grp & 1), (uint32_t)(cnt * chunks_all * 8));
        };
        if (collects) {
            arm_y(0);
            arm_y(1);
        }
        bool bad = false;
        const int seg_last = A.seg_last, segs_all = A.segs_all;
        const int carry = EXT ? A.carry : 0, nw = carry & 2 ? A.tail : nk;
        const uint32_t c_own = su32(sm + O.car) + (uint32_t)(tid * XF * 4);
        const uint32_t c_dst = carry & 2 ? peer_addr(c_own, (uint32_t)(A.base + rank + 1)) : 0u;
        const uint32_t c_bar = carry & 2 ? peer_addr(su32(bar_c), (uint32_t)(A.base + rank + 1)) : 0u;
        const unsigned long long new_item = A.new_item;
        // every part a partial sum of its own, or one row of them: one chain (with the
        // selects of the general case 24 parts took 1 230 cycles)
        const unsigned long long later = segs_all < 64 ? (1ull << segs_all) - 2ull : ~1ull;
        const bool flat = !SAME || new_item == later || new_item == 0ull;
        const uint32_t xbuf = (uint32_t)(Q.segs * Q.no_max * XF * 4);
        const uint32_t sbuf = (uint32_t)(Q.no_max * XF * 4);        // one part
        // the next phases are armed by a thread that has waited for the last ones
        bool arms = sub > 1 && wr == 0 && lane == 0;
        // A thread whose wait runs out keeps the common control flow, but waits for
        // nothing more, stores nothing into peers and arms nothing (a phase that it has
        // not seen complete must not be armed again).  So the peers' waits run out in
        // turn, after a step or two whose stores complete no phase.
        bool dead = false;
        auto wait = [&](uint64_t *b, uint32_t parity) {
            if (dead) return;
            for (int i = 0; !bar_try(b, parity);)
                if (__builtin_expect(++i >= Q.wait_limit, 0)) {
                    dead = true;
                    mon[0] = mon[1] = on = arms = false;
                    gave_up = 1;
                    break;
                }
        };
        // lane = 4 step + part: a quarter of the chunks' terms of one of eight steps
        auto collect = [&](int grp) {
            if (sub > 1) wait(bar_y + (grp & 1), (uint32_t)((grp >> 1) & 1));
            const int s8 = lane >> 2, part = lane & 3, n8 = grp * kPickSteps + s8;
            const float *pk = sm + O.pick + ((grp & 1) * kPickSteps + s8) * 2 * O.PS;
            float ys = 0.f, ye = 0.f;
            for (int j = part; j < sub * cmax; j += 4) {
                const float2 v = *reinterpret_cast<const float2 *>(pk + 2 * j);
                pickup_merge(ys, ye, v.x, v.y);
            }
#pragma unroll
            for (int o = 1; o <= 2; o <<= 1) {
                const float s2 = __shfl_xor_sync(0xffffffffu, ys, o);
                const float e2 = __shfl_xor_sync(0xffffffffu, ye, o);
                pickup_merge(ys, ye, s2, e2);
            }
            const float y = ys + ye;
            if (part == 0 && n8 < P.steps) {
                if ((!SAME || P.mode == MODE_FORWARD) && P.audio)
                    P.audio[(long long)A.plate * P.total_steps + P.n_begin + n8] = y;
                if (!isfinite(y)) bad = true;
            }
            if (!dead) arm_y(grp + 2);
        };
        bar_sync_id(1, WT);

        for (int it = 0; it < P.steps; ++it) {
            const bool rev_on = REV && it < rsteps;
            const bool rev_next = REV && it + 1 < rsteps;
            const int buf = it & 1;
            const int qb = REV ? buf * 4 * QB : 0;
            if (__builtin_expect((it & 31) == 0, 0)) load_block(it);
            // ---- row products, eta (xi, eta'), this warp's forces.  Rows and columns
            // beyond a class are zero, so nothing is guarded.
            float dot[R];
            if (kon) {
                const float *qs[R];
                qs[0] = qcol + qb;
                if constexpr (REV) qs[1] = qcol + bw;
                if constexpr (FUSED) qs[2] = qcol + br;
                float u[NR][R];
                if (SAME && !cls && N <= 32) {
#pragma unroll
                    for (int s = 0; s < NR; ++s)
#pragma unroll
                        for (int x = 0; x < R; ++x) u[s][x] = 0.f;
                    dense_row<R, NTM>(taddr, L, qs, u[0]);
                } else {
                    row_products<R, NTM, NSM, NREG, LMAX, (SAME || NR > 4 ? 1 : 2)>(hsm, WT, taddr, L, hreg, qs, u);
                }
                if constexpr (SAME)
#pragma unroll
                    for (int s = 0; s < NR; ++s)
#pragma unroll
                        for (int x = 0; x < R; ++x) fp[x * 4 * QB + gl * s] = u[s][x];
#pragma unroll
                for (int x = 0; x < R; ++x) dot[x] = 0.f;
                if (SAME && cls) {
                    // lane = column quad, the four row classes in order, as the streaming
                    // kernel's threads sum them
                    __syncwarp();
                    if (4 * lane < L)
#pragma unroll
                        for (int a = 0; a < 4; ++a) {
                            const int o = (a ^ kc) * QB + 4 * lane;
                            const float4 uv = *reinterpret_cast<const float4 *>(fpw + o);
                            const float4 qv = *reinterpret_cast<const float4 *>(rhs + qb + o);
                            dot[0] = fmaf(qv.w, uv.w, fmaf(qv.z, uv.z, fmaf(qv.y, uv.y, fmaf(qv.x, uv.x, dot[0]))));
                            if constexpr (REV) {
                                const float4 wv4 = *reinterpret_cast<const float4 *>(rhs + bw + o);
                                dot[1] = fmaf(wv4.w, uv.w, fmaf(wv4.z, uv.z, fmaf(wv4.y, uv.y, fmaf(wv4.x, uv.x, dot[1]))));
                            }
                            if constexpr (FUSED) {
                                const float4 rv = *reinterpret_cast<const float4 *>(rhs + br + o);
                                const float4 u2 = *reinterpret_cast<const float4 *>(fpw + 8 * QB + o);
                                dot[2] = fmaf(rv.w, u2.w, fmaf(rv.z, u2.z, fmaf(rv.y, u2.y, fmaf(rv.x, u2.x, dot[2]))));
                            }
                        }
                } else {
#pragma unroll
                    for (int s = 0; s < NR; ++s) {
                        dot[0] = fmaf(qrow[qb + gl * s], u[s][0], dot[0]);
                        if constexpr (REV) dot[1] = fmaf(qrow[bw + gl * s], u[s][0], dot[1]);
                        if constexpr (FUSED) dot[2] = fmaf(qrow[br + gl * s], u[s][2], dot[2]);
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int x = 0; x < R; ++x) dot[x] += __shfl_xor_sync(0xffffffffu, dot[x], o);
                if constexpr (!SAME) {
                    const float ke = kap * dot[0];
#pragma unroll
                    for (int s = 0; s < NR; ++s) fp[gl * s] = ke * u[s][0];
                } else if (lane == 0) {
                    float4 *const k4 = reinterpret_cast<float4 *>(kew + 8 * warp);
                    k4[0] = make_float4(kap * dot[0], kap, REV ? 2.f * dot[REV ? 1 : 0] : 0.f, dot[0]);
                    if constexpr (FUSED) k4[1] = make_float4(kap * dot[FUSED ? 2 : 0], 0.f, 0.f, 0.f);
                }
            }
            const float qn = REV ? rhs[qb + cpos] : 0.f;
            if (REV) copies_done();   // the next step's q^n (and this step's v^n) have arrived
            bar_sync_id(1, WT);       // the CTA's forces are in place, its right-hand sides read
            const int pb = (it / kPickSteps) & 1, ps = it % kPickSteps;
            // ---- forces.  A part is the sum over one run of stress modes, in order
            // (emit is called with each); the plate's force adds its parts in order,
            // item by item of the streaming kernel's work split where the plan asks
            // for its rounding (new_item), else all in one row.
            auto add_term = [&](int w, const float *p, float (&f)[R]) {
                const float4 k4 = *reinterpret_cast<const float4 *>(kew + 8 * w);
                const float uu = p[0];
                if constexpr (FWD) {
                    f[0] = fmaf(k4.x, uu, f[0]);
                } else {
                    f[1] = fmaf(k4.x, uu, f[1]);                                        // f(q^n)
                    f[0] = fmaf(k4.y, fmaf(k4.z, uu, k4.w * p[4 * QB]), f[0]);          // J w
                }
                if constexpr (FUSED) f[2] = fmaf(kew[8 * w + 4], p[8 * QB], f[2]);
            };
            auto parts = [&](int pos, float (&f)[R], auto emit) {      // f: where the first part stands
                const float *p = sm + O.fp + pos;
                if constexpr (!SAME) {
#pragma unroll
                    for (int w = 0; w < kResMaxWarps; ++w) f[0] += w < nk ? p[w * 4 * QB] : 0.f;
                    emit(0, f);
                    return;
                }
                int seg = 0;
#pragma unroll
                for (int w = 0; w < kResMaxWarps; ++w, p += R * 4 * QB) {
                    if (w >= nw) break;
                    add_term(w, p, f);
                    if (seg_last >> w & 1) {
                        emit(seg, f);
#pragma unroll
                        for (int x = 0; x < R; ++x) f[x] = 0.f;
                        ++seg;
                    }
                }
            };
            auto push_part = [&](uint32_t to, uint32_t bar, const float (&f)[R]) {
                if constexpr (R == 1) push1(to, bar, f[0]);
                if constexpr (R == 2) push2(to, bar, f[0], f[R - 1]);
                if constexpr (R == 3) push4(to, bar, f[0], f[R > 1 ? 1 : 0], f[R - 1]);
            };
            // a part that began in the CTA before goes on from there
            auto carried = [&](int h, float (&f)[R]) {
                const float *x = sm + O.car + (buf * Q.n_max + tid + h * WT) * XF;
#pragma unroll
                for (int y = 0; y < R; ++y) f[y] = x[y];
            };
            auto take_carry = [&]() {
                if (32 * warp < N) wait(bar_c, (uint32_t)buf);
                if (tid == 0 && !dead && it + 1 < P.steps) bar_expect_tx(bar_c, (uint32_t)(N * XF * 4));
            };
            float F[R], item[R];
#pragma unroll
            for (int x = 0; x < R; ++x) F[x] = item[x] = 0.f;
            auto add_part = [&](int g, const float (&v)[R]) {
                const bool fresh = SAME && (new_item >> g & 1);
#pragma unroll
                for (int x = 0; x < R; ++x) {
                    F[x] += fresh ? item[x] : 0.f;
                    item[x] = fresh ? v[x] : item[x] + v[x];
                }
            };
            auto load_part = [&](const float *x, float (&v)[R]) {
                if constexpr (R == 1) {
                    v[0] = x[0];
                } else if constexpr (R == 2) {
                    const float2 t = *reinterpret_cast<const float2 *>(x);
                    v[0] = t.x;
                    v[R - 1] = t.y;
                } else {
                    const float4 t = *reinterpret_cast<const float4 *>(x);
                    v[0] = t.x;
                    v[R > 1 ? 1 : 0] = t.y;
                    v[R - 1] = t.z;
                }
            };
            if (sub > 1) {
                if (EXT && carry != 0) {
                    // the part that ends in a later CTA first: the next one waits for it
                    const bool through = carry == 3 && nw == 0;
                    if (through) take_carry();
                    if (carry & 2) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (!mon[h]) continue;
                            float f[R];
#pragma unroll
                            for (int x = 0; x < R; ++x) f[x] = 0.f;
                            if (through) carried(h, f);
                            const float *p = sm + O.fp + mp[h] + nw * R * 4 * QB;
#pragma unroll 2
                            for (int w = nw; w < nk; ++w, p += R * 4 * QB) add_term(w, p, f);
                            push_part(c_dst + (uint32_t)((buf * Q.n_max + h * WT) * XF * 4), c_bar, f);
                        }
                    }
                    if ((carry & 1) && !through) take_carry();
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (!mon[h]) continue;
                    const uint32_t dst = mdst[h] + (buf ? xbuf : 0u);
                    float f[R];
#pragma unroll
                    for (int x = 0; x < R; ++x) f[x] = 0.f;
                    if (EXT && (carry & 1)) carried(h, f);
                    parts(mp[h], f, [&](int seg, const float (&v)[R]) { push_part(dst + seg * sbuf, mbar[h], v); });
                }
                if (upd) {
                    wait(bar_f, (uint32_t)buf);
                    const float *x = sm + O.xch + (buf * Q.segs * Q.no_max + oi) * XF;
                    if (on && flat) {
#pragma unroll 8
                        for (int g = 0; g < segs_all; ++g, x += Q.no_max * XF) {
                            float v[R];
                            load_part(x, v);
#pragma unroll
                            for (int y = 0; y < R; ++y) F[y] += v[y];
                        }
                    } else if (on) {
#pragma unroll 2
                        for (int g = 0; g < segs_all; ++g, x += Q.no_max * XF) {
                            float v[R];
                            load_part(x, v);
                            add_part(g, v);
                        }
                    }
                }
            } else if (on) {
                float f[R];
#pragma unroll
                for (int x = 0; x < R; ++x) f[x] = 0.f;
                parts(cpos, f, [&](int seg, const float (&v)[R]) { add_part(seg, v); });
            }
#pragma unroll
            for (int x = 0; x < R; ++x) F[x] += item[x];
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
                        const float x = REV ? wv : y0;
                        auto push_q = [&](uint32_t qa, uint32_t ba) {
                            push1(qa, ba, x);
                            if (FUSED) push1(qa + (uint32_t)((br - bw) * 4), ba, y0);
                        };
                        auto push_lays = [&](int pr, uint32_t qa, uint32_t ba) {
                            push_q(qa, ba);
                            if (more_lays) {
                                const int *row = dp + pr * Q.lays * Q.no_max + oi;
                                const int nl = row[0];
#pragma unroll 1
                                for (int l = 1; l < nl; ++l) push_q(qa + 4u * row[l * Q.no_max], ba);
                            }
                        };
                        push_lays(rep, q_dst0, q_bar0);
                        for (int pr = rep + reps; pr < sub; pr += reps)
                            push_lays(pr, peer_addr(q_dst, (uint32_t)(A.base + pr)),
                                      peer_addr(q_bar, (uint32_t)(A.base + pr)));
                    }
                } else {
                    if (on) {
                        if (FWD) rhs[cpos] = y0;
                        if (REV) rhs[bw + cpos] = wv;
                        if (FUSED) rhs[br + cpos] = y0;
                        if (more_lays)
#pragma unroll 1
                            for (int l = 1; l < lays; ++l) {
                                const int at = cpos + dp[l * Q.no_max + oi];
                                if (FWD) rhs[at] = y0;
                                if (REV) rhs[bw + at] = wv;
                                if (FUSED) rhs[br + at] = y0;
                            }
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
                // Kahan sums of x y, the product and the first subtraction in one rounding
                auto acc = [&](int idx, float x, float y) {
                    if (!(duty & (1 << idx))) return;
                    const float gs = ga[(2 * idx) * WT], gc = ga[(2 * idx + 1) * WT];
                    const float v = fmaf(x, y, -gc);
                    const float t = __fadd_rn(gs, v);
                    ga[(2 * idx) * WT] = t;
                    ga[(2 * idx + 1) * WT] = __fsub_rn(__fsub_rn(t, gs), v);
                };
                acc(GA_A, a_old, qn);
                acc(GA_V, a_old, sm[O.vst + tid]);
                acc(GA_F, a_old, fmaf(bcf, e, -F[R > 1 ? 1 : 0]));
                acc(GA_E, a_old, e);
                acc(GA_C, ybn, qn1);
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
            }
            if (FWD && picks) {
                float ys = 0.f, ye = 0.f;
                if (on) pickup_add(ys, ye, cw, cf[6 * WT], y0, y1);
                pst[ps * kPickPitch + lane] = make_float2(ys, ye);
                if (__builtin_expect(ps == kPickSteps - 1 || it == P.steps - 1, 0)) {
                    // the chunk's sums of up to eight steps, to the last rank
                    // (lane = 4 step + part, a quarter of the modes each)
                    __syncwarp();
                    const int s8 = lane >> 2, part = lane & 3;
                    ys = ye = 0.f;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float2 v = pst[s8 * kPickPitch + part + 4 * j];
                        pickup_merge(ys, ye, v.x, v.y);
                    }
#pragma unroll
                    for (int o = 1; o <= 2; o <<= 1) {
                        const float s2 = __shfl_xor_sync(0xffffffffu, ys, o);
                        const float e2 = __shfl_xor_sync(0xffffffffu, ye, o);
                        pickup_merge(ys, ye, s2, e2);
                    }
                    if (part == 0 && s8 <= ps && !dead) {
                        const int po = (pb * kPickSteps + s8) * 2 * O.PS;
                        if (sub > 1)
                            push2(y_dst0 + (uint32_t)(po * 4), y_bar0 + 8u * pb, ys, ye);
                        else
                            *reinterpret_cast<float2 *>(sm + O.pick + po + 2 * yent) = make_float2(ys, ye);
                    }
                }
            }
            // the last eight steps' samples, one step into the next eight
            if (collects && __builtin_expect(ps == 1 && it > kPickSteps, 0)) collect(it / kPickSteps - 1);
            if (ckpt && --ck_left == 0) {
                ck_left = P.ckpt_K;
                ++ck_idx;
            }
            wait(bar_q, (uint32_t)buf);
            if (arms && it + 1 < P.steps) bar_expect_tx(bar_q, tx_q);
        }

        // ---- the last samples, write back
        if (FWD) {
            bar_sync_id(1, WT);      // (one CTA: the terms of the last steps are in place)
            if (collects)
                for (int g = max(0, (P.steps - 2 - 1) / kPickSteps); g * kPickSteps < P.steps; ++g) {
                    // groups whose second next step never came
                    if (g * kPickSteps + kPickSteps + 1 < P.steps) continue;
                    collect(g);
                }
            if (__any_sync(0xffffffffu, bad) && lane == 0)
                set_status(P.status, A.plate, MDX_ERR_NONFINITE);
        }
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
        if (__any_sync(0xffffffffu, dead) && lane == 0) set_status(P.status, A.plate, MDX_ERR_TIMEOUT);
    }
    copies_done();
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem0), "r"(Q.tcols)
                     : "memory");
    // No peer stores into this CTA's shared memory from here on, and a CTA that waited for
    // everything sent to it has it.  Into one that gave up stores may still be on their
    // way, which no barrier counts to their end: it stays for far longer than their
    // hop of some 400 cycles.
    cluster_sync_all();
    if (gave_up)
        for (int i = 0; i < 64; ++i) __nanosleep(1000);
}

namespace {

// Kernel variants by longest row: a lane's rows in tensor memory (256 words a
// thread with more than four warps, else 512); of the others, those in registers
// (kernels without a reverse pass or checkpoints, NREG) and in shared memory.
constexpr int kVarLen[kResVariants] = {16, 24, 32, 40, 48, 56, 64, 64};
constexpr int kVarTm[kResVariants] = {2, 2, 4, 4, 4, 4, 4, 6};
constexpr int kVarSm[kResVariants] = {0, 1, 0, 1, 2, 3, 3, 2};
constexpr int kVarReg[kResVariants] = {0, 1, 0, 1, 2, 2, 0, 0};
int var_warps(int v) { return kVarTm[v] * kVarLen[v] > 256 ? 4 : kResMaxWarps; }
int var_sm(int v, bool same) { return kVarSm[v] - (same ? 0 : kVarReg[v]); }

template <int R, int ORD, int V>
const void *res_fn_v() {
    constexpr int REG = ORD > 0 ? 0 : kVarReg[V];
    return reinterpret_cast<const void *>(
        resident_kernel<R, kVarTm[V], kVarSm[V] - REG, REG, kVarLen[V], ORD>);
}

template <int R, int ORD>
const void *res_fn_r(int v) {
    switch (v) {
        case 0: return res_fn_v<R, ORD, 0>();
        case 1: return res_fn_v<R, ORD, 1>();
        case 2: return res_fn_v<R, ORD, 2>();
        case 3: return res_fn_v<R, ORD, 3>();
        case 4: return res_fn_v<R, ORD, 4>();
        case 5: return res_fn_v<R, ORD, 5>();
        case 6: return res_fn_v<R, ORD, 6>();
        default: return res_fn_v<R, ORD, 7>();
    }
}

// The kernel of r right-hand sides (passes with a reverse keep the streaming
// kernel's order, they have no other).
const void *res_fn(int r, const ResidentParams &Q) {
    const bool ext = Q.lays > 1 || Q.carry;
    if (r == 1) return !Q.same ? res_fn_r<1, 0>(Q.variant) : (ext ? res_fn_r<1, 2>(Q.variant) : res_fn_r<1, 1>(Q.variant));
    if (r == 2) return ext ? res_fn_r<2, 2>(Q.variant) : res_fn_r<2, 1>(Q.variant);
    return ext ? res_fn_r<3, 2>(Q.variant) : res_fn_r<3, 1>(Q.variant);
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
    const ResLayout o = res_layout(R, kVarLen[Q.variant], Q, var_sm(Q.variant, Q.same));
    return std::max(sizeof(float) * (size_t)o.end, (size_t)Q.tcols * kSmemPerColumn);
}

// Sets the kernels' attributes and returns how many clusters of cs CTAs run at
// once (0: the shape cannot be launched).
cudaError_t resident_check(int cs, const ResidentParams &Q, size_t smem_optin, int *fit) {
    *fit = 1 << 30;
    for (int r = 1; r <= (Q.same ? 3 : 1); ++r) {
        const void *fn = res_fn(r, Q);
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
        res_config(cfg, at, cs, cs, 32 * Q.warps, smem, nullptr);
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
    res_config(cfg, at, grid, cs, 32 * Q.warps, smem, s);
    ResidentParams q = Q;
    void *args[] = {&q};
    return cudaLaunchKernelExC(&cfg, res_fn(R, Q), args);
}

}  // namespace mdx
