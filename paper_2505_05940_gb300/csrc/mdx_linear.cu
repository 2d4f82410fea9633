// Linear modal response, parallel in time (Sec. 4.3.2).
//
// Without the nonlinear terms every mode obeys its own linear recursion
// (Sec. 3.2; Eq. 20-23 for Stormer-Verlet, Eq. 15-19 for the impulse-invariant
// scheme),
//     q^{n+1} = g q^n + p q^{n-1} + r b e^n,
// i.e. X^{n+1} = A X^n + (r b e^n, 0) with X^n = (q^n, q^{n-1}) and the
// companion matrix A = [[g, p], [1, 0]], whose eigenvalues are the discrete
// poles of the mode.  The paper evaluates such responses by repeated
// multiplication with the poles organised as a prefix scan over time; here
// the scan is blocked in time:
//   1. every chunk of L steps runs its inputs from a zero state (all chunks
//      and modes in parallel) and keeps only its final state E_j;
//   2. per mode, the chunk boundary states follow sequentially,
//      S_j = A^L S_{j-1} + E_j (A^L by repeated squaring, FP64), S_{-1} = X^0;
//   3. every chunk reruns from its true incoming state S_{j-1} and writes the
//      pickup y^n = sum_mu c_mu q_mu^{n+1}.
//
// Arithmetic.  The chunks' own responses, the chain over the chunks and the end
// states are FP64: a strongly damped mode's state leaves the range of FP32 within a
// chunk (eps reaches 1.2 for the upper modes of an ordinary plate).  Step 3 needs
// its states for FP32 samples only: it starts from the FP64 state and steps
// unevaluated FP32 pairs (about 48 bits) in the difference form (q, v = q - q^{n-1}),
// scaled per mode and chunk by a power of two to about 1 (its underflow is then
// below 2^-140 of the mode's largest value in the chunk).  The FP64 units do 2
// operations a cycle and SM, the FP32 units 128; a step costs 48 of the latter
// against 4 of the former.  The pickup's terms go through shared memory and each
// lane sums one step (shuffle sums of every step were the larger half of the
// time).  64 objects of 20 to 400 modes over 22 050 steps: 5.07 ms in FP64 throughout,
// 1.23 ms so (0.86 ms with step 1 in FP32 pairs too, which lost the end states of
// one mode in ten).
#include <cuda_runtime.h>

#include "../../include/mdx.h"
#include "mdx_common.cuh"
#include "mdx_scheme.cuh"

namespace mdx {

namespace {

constexpr int kLinThreads = 128;
constexpr int kLinWarps = kLinThreads / 32;

struct Pair {
    float h, l;
};

__device__ __forceinline__ Pair pair_of(double x) {
    Pair p;
    p.h = (float)x;
    p.l = (float)(x - (double)p.h);
    return p;
}

// (h, l) of a + b with |l| at most half an ulp of h, b any pair.
__device__ __forceinline__ Pair add(Pair a, Pair b) {
    const float s = a.h + b.h;
    const float bb = s - a.h;
    const float e = ((a.h - (s - bb)) + (b.h - bb)) + (a.l + b.l);
    Pair r;
    r.h = s + e;
    r.l = e - (r.h - s);
    return r;
}
// a b without renormalisation (the product's error in l).
__device__ __forceinline__ Pair mul(Pair a, Pair b) {
    Pair r;
    r.h = a.h * b.h;
    r.l = fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -r.h)));
    return r;
}

// Negated eps and rho, r b of a mode as pairs.
struct LinCoef {
    Pair neps, nrho, rb;
};

// The recursion's coefficients in FP64: q^{n+1} = g q^n + p q^{n-1} + rb e^n.
struct LinCoef64 {
    double g, p, rb;
};

__device__ __forceinline__ LinCoef64 lin_coef64(const LinearParams &P, long long gm) {
    const SchemeCoef k = scheme_coef(P.scheme, P.omega2[gm], P.gamma[gm], P.dt[gm]);
    LinCoef64 o;
    o.p = k.eps - 1.0;             // eps = 1 + p
    o.g = 2.0 - k.eps - k.rho;     // rho = 1 - g - p
    o.rb = k.r * P.b[gm];
    return o;
}

// v += r b e - eps v - rho q, q += v.
__device__ __forceinline__ void lin_step(const LinCoef &k, float e, Pair &q, Pair &v) {
    Pair u;
    u.h = k.rb.h * e;
    u.l = fmaf(k.rb.l, e, fmaf(k.rb.h, e, -u.h));
    v = add(v, add(add(mul(k.neps, v), u), mul(k.nrho, q)));
    q = add(q, v);
}

// Excitation of a chunk in shared memory (zeros without one).
template <typename T>
__device__ __forceinline__ void load_exc(const LinearParams &P, int inst, int n0, int n1, T *es) {
    const float *e = P.exc ? P.exc + (long long)inst * P.total_steps : nullptr;
    for (int n = n0 + threadIdx.x; n < n1; n += blockDim.x) es[n - n0] = e ? (T)e[n] : (T)0;
    __syncthreads();
}

// Largest magnitude of the chunk's excitation (NaN if there is one: its bits are the
// largest).
__device__ __forceinline__ float largest(const float *es, int cnt) {
    unsigned u = 0;
    for (int t = threadIdx.x & 31; t < cnt; t += 32) u = max(u, __float_as_uint(fabsf(es[t])));
    return __uint_as_float(__reduce_max_sync(0xffffffffu, u));
}

// A step is two FP64 operations: the response to e alone, r b applied at the end.
__global__ void __launch_bounds__(kLinThreads) lin_local_kernel(const LinearParams P) {
    __shared__ double es[kLinChunk];
    const int j = blockIdx.x, inst = blockIdx.y;
    if (j >= P.n_chunks - 1) return;        // the last chunk's end state is not needed
    const InstDesc d = P.inst[inst];
    const int n0 = j * P.L, n1 = min(P.steps, n0 + P.L);
    load_exc(P, inst, n0, n1, es);
    for (int m = threadIdx.x; m < d.N; m += kLinThreads) {
        const LinCoef64 k = lin_coef64(P, d.mode_off + m);
        double x0 = 0.0, x1 = 0.0;
#pragma unroll 4
        for (int n = 0; n < n1 - n0; ++n) {
            const double x = fma(k.g, x0, fma(k.p, x1, es[n]));
            x1 = x0;
            x0 = x;
        }
        double *E = P.E + ((long long)j * P.total_modes + d.mode_off + m) * 2;
        E[0] = k.rb * x0;
        E[1] = k.rb * x1;
    }
}

__global__ void lin_carry_kernel(const LinearParams P) {
    const long long gmode = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (gmode >= P.total_modes) return;
    const LinCoef64 k = lin_coef64(P, gmode);
    // A^L by repeated squaring
    double a00 = k.g, a01 = k.p, a10 = 1.0, a11 = 0.0;
    double r00 = 1.0, r01 = 0.0, r10 = 0.0, r11 = 1.0;
    for (int L = P.L; L > 0; L >>= 1) {
        if (L & 1) {
            const double t00 = r00 * a00 + r01 * a10, t01 = r00 * a01 + r01 * a11;
            const double t10 = r10 * a00 + r11 * a10, t11 = r10 * a01 + r11 * a11;
            r00 = t00, r01 = t01, r10 = t10, r11 = t11;
        }
        const double s00 = a00 * a00 + a01 * a10, s01 = a00 * a01 + a01 * a11;
        const double s10 = a10 * a00 + a11 * a10, s11 = a10 * a01 + a11 * a11;
        a00 = s00, a01 = s01, a10 = s10, a11 = s11;
    }
    double s0 = P.q0 ? P.q0[gmode] : 0.0, s1 = P.qm1 ? P.qm1[gmode] : 0.0;
    const long long st = P.total_modes * 2;
    double *S = P.S + gmode * 2;
    S[0] = s0;
    S[1] = s1;
    // the next chunks' end states are loaded together, ahead of the chain
    constexpr int U = 8;
    for (int j0 = 0; j0 < P.n_chunks - 1; j0 += U) {
        double e0[U], e1[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool in = j0 + u < P.n_chunks - 1;
            const double *E = P.E + (long long)(j0 + u) * st + gmode * 2;
            e0[u] = in ? E[0] : 0.0;
            e1[u] = in ? E[1] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (j0 + u >= P.n_chunks - 1) break;
            const double t0 = fma(r00, s0, fma(r01, s1, e0[u]));
            s1 = fma(r10, s0, fma(r11, s1, e1[u]));
            s0 = t0;
            double *Sj = P.S + (long long)(j0 + u + 1) * st + gmode * 2;
            Sj[0] = s0;
            Sj[1] = s1;
        }
    }
}

// End states of an instance: its last chunk from its true incoming state, FP64.
__device__ void end_states(const LinearParams &P, int inst, float *es) {
    const InstDesc d = P.inst[inst];
    const int j = P.n_chunks - 1, n0 = j * P.L, cnt = P.steps - n0;
    load_exc(P, inst, n0, P.steps, es);
    for (int m = threadIdx.x; m < d.N; m += kLinThreads) {
        const long long gm = d.mode_off + m;
        const LinCoef64 k = lin_coef64(P, gm);
        const double *S = P.S + ((long long)j * P.total_modes + gm) * 2;
        double x0 = S[0], x1 = S[1];
#pragma unroll 4
        for (int n = 0; n < cnt; ++n) {
            const double x = fma(k.g, x0, fma(k.p, x1, k.rb * (double)es[n]));
            x1 = x0;
            x0 = x;
        }
        if (P.q_end) P.q_end[gm] = x0;
        if (P.qm1_end) P.qm1_end[gm] = x1;
    }
}

// Blocks: the instances' end states if asked for, then every (chunk, instance).
__global__ void __launch_bounds__(kLinThreads) lin_out_kernel(const LinearParams P) {
    __shared__ float es[kLinChunk];
    __shared__ float2 terms[kLinWarps][32][33];       // [step][mode], rows without conflicts
    __shared__ float2 ypart[kLinWarps][kLinChunk];
    unsigned blk = blockIdx.x;
    if (P.q_end || P.qm1_end) {
        if (blk < (unsigned)P.n_inst) {
            end_states(P, (int)blk, es);
            return;
        }
        blk -= P.n_inst;
    }
    const int inst = (int)(blk % P.n_inst), j = (int)(blk / P.n_inst);
    const InstDesc d = P.inst[inst];
    const int n0 = j * P.L, cnt = min(P.steps, n0 + P.L) - n0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int t = lane; t < kLinChunk; t += 32) ypart[warp][t] = make_float2(0.f, 0.f);
    load_exc(P, inst, n0, n0 + cnt, es);
    const float emax = largest(es, cnt);
    // every warp walks whole rounds of 32 modes
    for (int m0 = warp * 32; m0 < d.N; m0 += kLinThreads) {
        const int m = m0 + lane;
        const bool on = m < d.N;
        const long long gm = d.mode_off + m;
        LinCoef k = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
        Pair q = {0.f, 0.f}, v = {0.f, 0.f}, c = {0.f, 0.f};
        if (on) {
            const SchemeCoef sc = scheme_coef(P.scheme, P.omega2[gm], P.gamma[gm], P.dt[gm]);
            const double *S = P.S + ((long long)j * P.total_modes + gm) * 2;
            const double q0 = S[0], v0 = S[0] - S[1], rb = sc.r * P.b[gm];
            // the scale 2^x: state and input to about 1 (r b stays an FP32 number where
            // the whole input is tiny), its inverse in the pickup weight
            const double big = fmax(fmax(fabs(q0), fabs(v0)), fabs(rb) * (double)emax);
            int x = 0;
            if (big > 0.0 && isfinite(big)) {
                x = -ilogb(big);
                if (rb != 0.0) x = min(x, 120 - ilogb(rb));
            }
            k.neps = pair_of(-sc.eps);
            k.nrho = pair_of(-sc.rho);
            k.rb = pair_of(scalbn(rb, x));
            q = pair_of(scalbn(q0, x));
            v = pair_of(scalbn(v0, x));
            c = pair_of(scalbn(P.c[gm], -x));
        }
        const int modes = min(32, d.N - m0);
        for (int i0 = 0; i0 < cnt; i0 += 32) {
            const int ni = min(32, cnt - i0);
#pragma unroll 4
            for (int i = 0; i < ni; ++i) {
                lin_step(k, es[i0 + i], q, v);
                float ys = 0.f, ye = 0.f;
                pickup_add(ys, ye, c.h, c.l, q.h, q.l);
                terms[warp][i][lane] = make_float2(ys, ye);
            }
            __syncwarp();
            // lane l sums the modes of step i0 + l
            if (lane < ni) {
                float2 y = ypart[warp][i0 + lane];
#pragma unroll 8
                for (int q2 = 0; q2 < modes; ++q2) {
                    const float2 t = terms[warp][lane][q2];
                    pickup_merge(y.x, y.y, t.x, t.y);
                }
                ypart[warp][i0 + lane] = y;
            }
            __syncwarp();
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < cnt; t += kLinThreads) {
        float ys = 0.f, ye = 0.f;
#pragma unroll
        for (int w = 0; w < kLinWarps; ++w) pickup_merge(ys, ye, ypart[w][t].x, ypart[w][t].y);
        const float y = (float)((double)ys + (double)ye);
        if (P.audio) P.audio[(long long)inst * P.total_steps + n0 + t] = y;
        if (!isfinite(y)) set_status(P.status, inst, MDX_ERR_NONFINITE);
    }
}

}  // namespace

cudaError_t launch_linear(const LinearParams &P, cudaStream_t s) {
    if (P.steps <= 0 || P.n_inst <= 0) return cudaSuccess;
    const dim3 grid(P.n_chunks, P.n_inst);
    lin_local_kernel<<<grid, kLinThreads, 0, s>>>(P);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int cb = 128;
    lin_carry_kernel<<<(int)((P.total_modes + cb - 1) / cb), cb, 0, s>>>(P);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long blocks = (P.n_chunks + (P.q_end || P.qm1_end ? 1LL : 0LL)) * P.n_inst;
    lin_out_kernel<<<(unsigned)blocks, kLinThreads, 0, s>>>(P);
    return cudaGetLastError();
}

}  // namespace mdx
