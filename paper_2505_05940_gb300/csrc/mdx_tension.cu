// Strings (Kirchhoff-Carrier) and membranes (Berger): one warp per instance of up
// to 128 modes, 2 to 8 warps (128 modes each) above.
//
// Per step (Sec. 3.2, Eq. 20 in difference form; Sec. 3.1, Eq. 8):
//   S       = sum_nu lambda_nu q_nu^2                      (warp reduction)
//   fnl_mu  = tau' lambda_mu q_mu S
//   v, q    <- Stormer-Verlet difference-form update
//   y^n     = sum_mu c_mu q^{n+1}_mu
// Lane l holds modes l, l + 32, ...; the whole time loop runs inside the kernel
// with the state in registers.  The
// same kernel re-runs a segment from a checkpoint (storing every state) and
// sweeps a stored segment backwards (adjoint recursion, J symmetric because
// fnl = grad V, V = tau'/4 S^2).
//
// Bound: the dependent chain of a step (update, lambda q^2, the shuffles of S),
// so everything else is kept off it.  The pickup's terms go to shared memory
// and are summed once per 32 steps, one step per lane (two interleaved
// reductions per step took 410 cycles a step for 40 modes, this 290); the
// reverse sweep's states arrive by asynchronous copies, a block of steps ahead
// (a fit's step of 48 strings of 40 to 100 modes, forward, recompute and
// reverse over 4 410 steps, took 5.6 ms with loads inside the step, now 3.6 ms).
#include <cuda_runtime.h>

#include <algorithm>

#include "../../include/mdx.h"
#include "mdx_common.cuh"

namespace mdx {

namespace {

constexpr int kPickRow = 33;     // pickup row stride (float2): lanes read rows without conflicts

__device__ __forceinline__ void copy4(float *dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Steps per staged block of the reverse sweep: two buffers of (q, v) rows.
__host__ __device__ constexpr int rev_block(int J) { return J <= 2 ? 16 : 8; }

}  // namespace

// Sums over the instance: the lanes, then the warps in order (through
// shared memory, double-buffered by step: one barrier).
template <int W, int V>
__device__ __forceinline__ void instance_sum(float (&v)[V], float (*red)[V][W], int parity, int warp) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int x = 0; x < V; ++x) v[x] += __shfl_xor_sync(0xffffffffu, v[x], o);
    if constexpr (W > 1) {
        if ((threadIdx.x & 31) == 0)
#pragma unroll
            for (int x = 0; x < V; ++x) red[parity][x][warp] = v[x];
        __syncthreads();
#pragma unroll
        for (int x = 0; x < V; ++x) {
            v[x] = red[parity][x][0];
#pragma unroll
            for (int w = 1; w < W; ++w) v[x] += red[parity][x][w];
        }
    }
}

template <int J, int W, bool REV>
__global__ void __launch_bounds__(32 * W) tension_kernel(const TensionParams P) {
    // per warp: forward pickup terms [32][kPickRow] x 2; reverse [2][U][2][32 J]
    extern __shared__ __align__(16) float tsm_all[];
    __shared__ float red[2][REV ? 2 : 1][W];
    __shared__ float2 ypart[W][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *tsm = tsm_all + warp * (REV ? 2 * rev_block(J) * 2 * 32 * J : 2 * 32 * kPickRow);
    const int inst = P.list[blockIdx.x];
    const InstDesc d = P.inst[inst];
    const int N = d.N;
    const long long mo = d.mode_off;
    const long long TM = P.total_modes;
    const float taup = d.taup;
    const int l0 = lane + warp * 32 * J;

    float eps[J], rw2[J], rw2l[J], r[J], b[J], c[J], clo[J], lam[J];
    float x0[J], x1[J], x2[J], x3[J];   // forward: q_hi, q_lo, v_hi, v_lo ; reverse: a_hi, a_lo, mu
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int m = l0 + 32 * j;
        const bool ok = m < N;
        eps[j] = ok ? P.coef.eps[mo + m] : 0.f;
        rw2[j] = ok ? P.coef.rw2[mo + m] : 0.f;
        rw2l[j] = ok ? P.coef.rw2lo[mo + m] : 0.f;
        r[j] = ok ? P.coef.r[mo + m] : 0.f;
        b[j] = ok ? P.coef.b[mo + m] : 0.f;
        c[j] = ok ? P.coef.c[mo + m] : 0.f;
        clo[j] = ok ? P.coef.clo[mo + m] : 0.f;
        lam[j] = ok ? P.coef.lam[mo + m] : 0.f;
    }
    const float *exc = P.exc ? P.exc + (long long)inst * P.total_steps : nullptr;

    if constexpr (!REV) {
        // ---------------------------------------------------------- forward / recompute
        float2 *pk = reinterpret_cast<float2 *>(tsm);
        const float *src = P.state_io;
        if (P.mode == MODE_RECOMPUTE) src = P.ckpt + (long long)(P.n_begin / P.ckpt_K) * kStateArrays * TM;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int m = l0 + 32 * j;
            const bool ok = m < N;
            x0[j] = ok ? src[mo + m] : 0.f;
            x1[j] = ok ? src[TM + mo + m] : 0.f;
            x2[j] = ok ? src[2 * TM + mo + m] : 0.f;
            x3[j] = ok ? src[3 * TM + mo + m] : 0.f;
        }
        float S[1] = {0.f};
#pragma unroll
        for (int j = 0; j < J; ++j) S[0] = fmaf(lam[j] * x0[j], x0[j], S[0]);
        instance_sum<W, 1>(S, red, 1, warp);
        float *aud = P.audio ? P.audio + (long long)inst * P.total_steps : nullptr;
        const bool rec = P.mode == MODE_RECOMPUTE;
        const bool ckpt = P.mode == MODE_FORWARD && P.ckpt;
        float *ck = ckpt ? P.ckpt + mo : nullptr;
        float *sq = rec ? P.seg_q + mo : nullptr, *sv = rec ? P.seg_v + mo : nullptr;
        bool bad = false;
        auto store2 = [&](float *dq, float *dv) {
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int m = l0 + 32 * j;
                if (m < N) {
                    dq[m] = x0[j];
                    dv[m] = x2[j];
                }
            }
        };
        // one step; the pickup's terms go to row i
        int par = 0;
        auto step = [&](int i, float e) {
            float Sp[1] = {0.f};
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const float f = taup * lam[j] * x0[j] * S[0];
                sv_step(x0[j], x1[j], x2[j], x3[j], eps[j], rw2[j], rw2l[j], r[j], fmaf(b[j], e, -f));
                Sp[0] = fmaf(lam[j] * x0[j], x0[j], Sp[0]);
            }
            instance_sum<W, 1>(Sp, red, par, warp);
            S[0] = Sp[0];
            par ^= 1;
            // the first mode's term starts the compensated sum
            float ys = c[0] * x0[0];
            float ye = fmaf(c[0], x1[0], fmaf(clo[0], x0[0], fmaf(c[0], x0[0], -ys)));
#pragma unroll
            for (int j = 1; j < J; ++j) pickup_add(ys, ye, c[j], clo[j], x0[j], x1[j]);
            pk[i * kPickRow + lane] = make_float2(ys, ye);
        };
        auto load_e = [&](int i) {
            return (exc && i + lane < P.steps) ? exc[P.n_begin + i + lane] : 0.f;
        };
        // blocks of at most 32 steps that end at the checkpoints
        int ck_left = 0;
        float enext = load_e(0);
        for (int i0 = 0; i0 < P.steps;) {
            int cnt = min(32, P.steps - i0);
            if (ckpt) {
                if (ck_left == 0) {
                    ck_left = P.ckpt_K;
                    store2(ck, ck + 2 * TM);
#pragma unroll
                    for (int j = 0; j < J; ++j) {
                        const int m = l0 + 32 * j;
                        if (m < N) {
                            ck[TM + m] = x1[j];
                            ck[3 * TM + m] = x3[j];
                        }
                    }
                    ck += (long long)kStateArrays * TM;
                }
                cnt = min(cnt, ck_left);
                ck_left -= cnt;
            }
            const float ebuf = enext;
            enext = load_e(i0 + cnt);
            if (rec) {
#pragma unroll 2
                for (int i = 0; i < cnt; ++i) {
                    store2(sq, sv);
                    sq += TM;
                    sv += TM;
                    step(i, __shfl_sync(0xffffffffu, ebuf, i));
                }
            } else {
#pragma unroll 4
                for (int i = 0; i < cnt; ++i) step(i, __shfl_sync(0xffffffffu, ebuf, i));
            }
            __syncwarp();
            // lane l sums the terms of step i0 + l
            float ys = 0.f, ye = 0.f;
#pragma unroll 8
            for (int k = 0; k < 32; ++k) {
                const float2 v = pk[lane * kPickRow + k];
                pickup_merge(ys, ye, v.x, v.y);
            }
            if constexpr (W > 1) {
                ypart[warp][lane] = make_float2(ys, ye);
                __syncthreads();
#pragma unroll
                for (int w = 1; w < W; ++w)
                    if (warp == 0) pickup_merge(ys, ye, ypart[w][lane].x, ypart[w][lane].y);
            }
            if (lane < cnt && warp == 0) {
                const float y = ys + ye;
                if (aud) aud[P.n_begin + i0 + lane] = y;
                if (!isfinite(y)) bad = true;
            }
            __syncwarp();
            i0 += cnt;
        }
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int m = l0 + 32 * j;
            if (m >= N) continue;
            if (rec) {
                sq[m] = x0[j];
                sv[m] = x2[j];
            } else {
                P.state_io[mo + m] = x0[j];
                P.state_io[TM + mo + m] = x1[j];
                P.state_io[2 * TM + mo + m] = x2[j];
                P.state_io[3 * TM + mo + m] = x3[j];
            }
        }
        bad = __any_sync(0xffffffffu, bad);
        if (bad && lane == 0) set_status(P.status, inst, MDX_ERR_NONFINITE);
    } else {
    // ------------------------------------------------------------------ reverse sweep
    // seg_q[t], seg_v[t] hold q^{n0+t}, v^{n0+t} for t = 0..steps.
    constexpr int U = rev_block(J);
    float q1[J];                        // q^{n+1}
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int m = l0 + 32 * j;
        const bool ok = m < N;
        x0[j] = ok ? P.adj[mo + m] : 0.f;
        x1[j] = ok ? P.adj[TM + mo + m] : 0.f;
        x2[j] = ok ? P.adj[2 * TM + mo + m] : 0.f;
        q1[j] = ok ? P.seg_q[(long long)P.steps * TM + mo + m] : 0.f;
    }
    float gs[GA_N][J], gc[GA_N][J];
#pragma unroll
    for (int g = 0; g < GA_N; ++g)
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int m = l0 + 32 * j;
            const bool ok = m < N;
            gs[g][j] = ok ? P.gacc[(long long)(2 * g) * TM + mo + m] : 0.f;
            gc[g][j] = ok ? P.gacc[(long long)(2 * g + 1) * TM + mo + m] : 0.f;
        }
    float ts = 0.f, tc = 0.f;
    if (threadIdx.x == 0) { ts = P.tacc[2 * inst]; tc = P.tacc[2 * inst + 1]; }
    const float *yb = P.ybar + (long long)inst * P.total_steps;
    bool bad = false;
    // block k: local steps t = steps - 1 - k U - u, u = 0 .. U - 1
    auto stage = [&](int k) {
        float *buf = tsm + (k & 1) * (U * 2 * 32 * J);
        for (int u = 0; u < U; ++u) {
            const int t = P.steps - 1 - k * U - u;
            if (t < 0) break;
            const float *sq = P.seg_q + (long long)t * TM + mo, *sv = P.seg_v + (long long)t * TM + mo;
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int m = l0 + 32 * j;
                float *dst = buf + (u * 2 * J + j) * 32 + lane;
                if (m < N) {
                    copy4(dst, sq + m);
                    copy4(dst + 32 * J, sv + m);
                }
            }
        }
    };
    for (int e = lane; e < 2 * U * 2 * 32 * J; e += 32) tsm[e] = 0.f;   // lanes beyond N read zeros
    stage(0);
    // targets and excitation: a lane holds one of 32 steps
    float ebuf = 0.f, ybuf = 0.f;
    float ybn = P.steps > 0 ? yb[P.n_begin + P.steps - 1] : 0.f;
    for (int k = 0; k * U < P.steps; ++k) {
        copies_done();                  // each lane reads only what it copied
        if ((k + 1) * U < P.steps) stage(k + 1);
        const float *buf = tsm + (k & 1) * (U * 2 * 32 * J);
#pragma unroll 1
        for (int u = 0; u < U; ++u) {
            const int s = k * U + u;
            if (s >= P.steps) break;
            if ((s & 31) == 0) {
                const int tl = P.steps - 1 - s - lane, nl = P.n_begin + tl;
                ebuf = (exc && tl >= 0) ? exc[nl] : 0.f;
                ybuf = (tl >= 0 && nl >= 1) ? yb[nl - 1] : 0.f;
            }
            const float e = __shfl_sync(0xffffffffu, ebuf, s & 31);
            const float ybm = __shfl_sync(0xffffffffu, ybuf, s & 31);
            float q[J], wv[J];
            float SP[2] = {0.f, 0.f};
#pragma unroll
            for (int j = 0; j < J; ++j) {
                q[j] = buf[(u * 2 * J + j) * 32 + lane];
                wv[j] = r[j] * x0[j];
                SP[0] = fmaf(lam[j] * q[j], q[j], SP[0]);
                SP[1] = fmaf(lam[j] * q[j], wv[j], SP[1]);
            }
            instance_sum<W, 2>(SP, red, s & 1, warp);
            const float S = SP[0], Pq = SP[1];
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const float a = x0[j];
                const float f = taup * lam[j] * q[j] * S;
                const float Jw = taup * lam[j] * fmaf(S, wv[j], 2.f * q[j] * Pq);
                adj_step(x0[j], x1[j], x2[j], eps[j], rw2[j], Jw, c[j] * ybm);
                const float v = buf[(u * 2 * J + J + j) * 32 + lane];
                kahan_add(gs[GA_A][j], gc[GA_A][j], a * q[j]);
                kahan_add(gs[GA_V][j], gc[GA_V][j], a * v);
                kahan_add(gs[GA_F][j], gc[GA_F][j], a * fmaf(b[j], e, -f));
                kahan_add(gs[GA_E][j], gc[GA_E][j], a * e);
                kahan_add(gs[GA_C][j], gc[GA_C][j], ybn * q1[j]);
                q1[j] = q[j];
            }
            ybn = ybm;
            if (threadIdx.x == 0) kahan_add(ts, tc, -S * Pq);
            if (!isfinite(x0[0])) bad = true;
        }
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int m = l0 + 32 * j;
        if (m < N) {
            P.adj[mo + m] = x0[j];
            P.adj[TM + mo + m] = x1[j];
            P.adj[2 * TM + mo + m] = x2[j];
#pragma unroll
            for (int g = 0; g < GA_N; ++g) {
                P.gacc[(long long)(2 * g) * TM + mo + m] = gs[g][j];
                P.gacc[(long long)(2 * g + 1) * TM + mo + m] = gc[g][j];
            }
        }
    }
    if (threadIdx.x == 0) { P.tacc[2 * inst] = ts; P.tacc[2 * inst + 1] = tc; }
    if (bad && lane == 0) set_status(P.status, inst, MDX_ERR_NONFINITE);
    }
}

template <int J, int W>
static cudaError_t launch_j(const TensionParams &p, cudaStream_t s) {
    if (p.n_list == 0) return cudaSuccess;
    if (p.mode == MODE_REVERSE) {
        const size_t smem = sizeof(float) * W * 2 * rev_block(J) * 2 * 32 * J;
        if (smem > 48 * 1024) {
            const cudaError_t e = cudaFuncSetAttribute(
                tension_kernel<J, W, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        tension_kernel<J, W, true><<<p.n_list, 32 * W, smem, s>>>(p);
    } else {
        const size_t smem = sizeof(float) * W * 2 * 32 * kPickRow;
        if (smem > 48 * 1024) {
            const cudaError_t e = cudaFuncSetAttribute(
                tension_kernel<J, W, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        tension_kernel<J, W, false><<<p.n_list, 32 * W, smem, s>>>(p);
    }
    return cudaGetLastError();
}

// Modes per lane and warps, by the largest instance: each further mode of a lane
// adds about 35 instructions to a step; above four a further warp costs less (a
// barrier and a shared-memory sum, about 90 cycles, against 140).
cudaError_t launch_tension(const TensionParams &p, int max_n, cudaStream_t s) {
    if (max_n <= 32) return launch_j<1, 1>(p, s);
    if (max_n <= 64) return launch_j<2, 1>(p, s);
    if (max_n <= 96) return launch_j<3, 1>(p, s);
    if (max_n <= 128) return launch_j<4, 1>(p, s);
    if (max_n <= 256) return launch_j<4, 2>(p, s);
    if (max_n <= 512) return launch_j<4, 4>(p, s);
    return launch_j<4, 8>(p, s);
}

}  // namespace mdx
