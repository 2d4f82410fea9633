// Log-mel features of simulated audio: the input of the learned proposal
// network (initial estimates for the inverse fits of Sec. 4.3).
//
// Per signal x of length T and segment s of S:
//   frames   f = 0 .. F-1, F = 1 + T / hop, frame f covers the signal extended
//            by reflection by n_fft / 2 on both sides (centred frames), times
//            the periodic Hann window w_j = (1 - cos(2 pi j / n_fft)) / 2;
//   power    P_f[k] = |sum_j w_j x_f[j] e^{-2 pi i j k / n_fft}|^2, k <= n_fft / 2;
//   mel      m_f[i] = log(sum_k W[i][k] P_f[k] + 1e-6), W the triangular filters
//            equally spaced on the HTK mel scale mel(f) = 2595 log10(1 + f / 700)
//            between fmin and fmax (n_mels + 2 points; filter i rises from
//            point i to point i+1 and falls to point i+2);
//   output   out[i][s] = mean of m_f[i] over frames floor(s F / S) .. floor((s+1) F / S) - 1
//            (at least one frame).
// The real FFT of a frame is the complex FFT of its even and odd samples (half
// the length, so rounding stays within the frame), radix-4 Stockham passes in
// shared memory, then the split into the spectrum of the frame.  Everything a
// call's frames share (window, twiddles, filter weights, from FP64) is built
// once per CTA, and the CTAs are persistent: FP64 runs at 1/64 of the FP32 rate
// here, and building the tables and the window per (segment, signal), with a
// cospi per sample and frame, took most of the 4.5 ms of 1 024 signals of
// 11 025 samples (now 0.38 ms; the frames' passes through shared memory bound it).  A
// CTA is four groups of 256 threads; a group works on one (segment, signal) at
// a time, two frames at once, the frames in order: the result is deterministic.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "../../include/mdx.h"
#include "mdx_internal.h"

namespace mdx {

namespace {

constexpr int kFeatGroups = 4;               // independent groups of a CTA at most
constexpr int kFeatThreads = 256;            // threads of a group
constexpr int kFeatMaxMels = 512;

struct LogmelArgs {
    const float *audio;
    int batch, T, n_fft, log2m, hop, n_mels, segments, groups;   // log2m: of n_fft / 2
    double fs, fmin, fmax;
    float *out;
};

__device__ __forceinline__ double hz_to_mel(double f) { return 2595.0 * log10(1.0 + f / 700.0); }
__device__ __forceinline__ double mel_to_hz(double m) { return 700.0 * (exp10(m / 2595.0) - 1.0); }

// Padded place of element i of an FFT buffer: one extra element every 16, so that
// the first pass's stride-4 stores do not collide.
__host__ __device__ __forceinline__ int fpad(int i) { return i + (i >> 4); }

// Byte offsets of the shared-memory arrays (one definition for the kernel and
// the launch): tables, then per group X [2 buffers][2 frames], P [2 frames].
struct FeatLayout {
    size_t tw, win, w1, w2, cut, pts, group, X, P, acc, group_bytes;
};

__host__ __device__ inline FeatLayout feat_layout(int n_fft, int n_mels) {
    const size_t m = (size_t)n_fft / 2;
    FeatLayout L;
    L.tw = 0;                                               // [n] float2
    L.win = L.tw + sizeof(float2) * (size_t)n_fft;          // [n]
    L.w1 = L.win + sizeof(float) * (size_t)n_fft;           // [m + 1] falling edge
    L.w2 = L.w1 + sizeof(float) * (m + 1);                  // [m + 1] rising edge
    L.cut = L.w2 + sizeof(float) * (m + 1);                 // [n_mels + 3] first bin above a point
    L.pts = (L.cut + sizeof(int) * (size_t)(n_mels + 3) + 7) & ~(size_t)7;   // [n_mels + 2]
    L.group = (L.pts + sizeof(double) * (size_t)(n_mels + 2) + 15) & ~(size_t)15;
    L.X = 0;
    L.P = sizeof(float2) * 4 * (size_t)(fpad((int)m) + 1);
    L.acc = L.P + sizeof(float) * 2 * (m + 1);
    L.group_bytes = (L.acc + sizeof(float) * 2 * (size_t)n_mels + 15) & ~(size_t)15;
    return L;
}

__device__ __forceinline__ void group_bar(int g) {
    asm volatile("barrier.sync %0, %1;" ::"r"(g + 1), "n"(kFeatThreads) : "memory");
}

__device__ __forceinline__ float2 cmul(float2 a, float2 w) {
    return make_float2(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x);
}

// One radix-4 butterfly (forward transform).
__device__ __forceinline__ void fft4(float2 (&v)[4]) {
    const float2 a = make_float2(v[0].x + v[2].x, v[0].y + v[2].y);
    const float2 b = make_float2(v[0].x - v[2].x, v[0].y - v[2].y);
    const float2 c = make_float2(v[1].x + v[3].x, v[1].y + v[3].y);
    const float2 d = make_float2(v[1].y - v[3].y, v[3].x - v[1].x);   // -i (v1 - v3)
    v[0] = make_float2(a.x + c.x, a.y + c.y);
    v[1] = make_float2(b.x + d.x, b.y + d.y);
    v[2] = make_float2(a.x - c.x, a.y - c.y);
    v[3] = make_float2(b.x - d.x, b.y - d.y);
}

__global__ void __launch_bounds__(kFeatGroups *kFeatThreads, 1) logmel_kernel(const LogmelArgs A) {
    extern __shared__ __align__(16) unsigned char fsm[];
    const int n = A.n_fft, m = n / 2, nm = A.n_mels;
    const FeatLayout FL = feat_layout(n, nm);
    float2 *tw = reinterpret_cast<float2 *>(fsm + FL.tw);
    float *win = reinterpret_cast<float *>(fsm + FL.win);
    float *w1 = reinterpret_cast<float *>(fsm + FL.w1);
    float *w2 = reinterpret_cast<float *>(fsm + FL.w2);
    int *cut = reinterpret_cast<int *>(fsm + FL.cut);
    double *pts = reinterpret_cast<double *>(fsm + FL.pts);
    const int T = A.T, hop = A.hop, S = A.segments;
    const int F = 1 + T / hop;

    // ---- tables.  Twiddles e^{-2 pi i k / n} and the window by symmetry from the
    // first octant's FP64 values
    for (int t = threadIdx.x; t <= n / 8; t += blockDim.x) {
        double sn, cs;
        sincospi(2.0 * t / n, &sn, &cs);
        const float c = (float)cs, s = (float)sn;
        const int q = n / 4;
        tw[t] = make_float2(c, -s);
        tw[q - t] = make_float2(s, -c);
        tw[q + t] = make_float2(-s, -c);
        tw[2 * q - t] = make_float2(-c, -s);
        tw[2 * q + t] = make_float2(-c, s);
        tw[3 * q - t] = make_float2(-s, c);
        tw[3 * q + t] = make_float2(s, c);
        if (t > 0) tw[n - t] = make_float2(c, s);
        const float wa = (float)(0.5 * (1.0 - cs)), wb = (float)(0.5 * (1.0 - sn));
        const float wc = (float)(0.5 * (1.0 + sn)), wd = (float)(0.5 * (1.0 + cs));
        win[t] = wa;
        win[q - t] = wb;
        win[q + t] = wc;
        win[2 * q - t] = wd;
        win[2 * q + t] = wd;
        win[3 * q - t] = wc;
        win[3 * q + t] = wb;
        if (t > 0) win[n - t] = wa;
    }
    // mel points (numpy linspace: a + j step, the last point exact)
    const double m_lo = hz_to_mel(A.fmin), m_hi = hz_to_mel(A.fmax);
    const double mstep = (m_hi - m_lo) / (nm + 1);
    for (int j = threadIdx.x; j < nm + 2; j += blockDim.x)
        pts[j] = mel_to_hz(j == nm + 1 ? m_hi : m_lo + j * mstep);
    for (int j = threadIdx.x; j < nm + 3; j += blockDim.x) cut[j] = m + 1;
    __syncthreads();
    // per bin: the largest j with pts[j] < f; it lies on the falling edge of
    // triangle j - 1 and on the rising edge of triangle j
    const double df = (A.fs / 2.0) / m;
    auto point_below = [&](int k) {
        const double f = (k == m) ? A.fs / 2.0 : k * df;
        int lo = -1, hi = nm + 2;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (pts[mid] < f) lo = mid; else hi = mid;
        }
        return lo;
    };
    for (int k = threadIdx.x; k <= m; k += blockDim.x) {
        const double f = (k == m) ? A.fs / 2.0 : k * df;
        const int j = point_below(k), jp = k > 0 ? point_below(k - 1) : -1;
        for (int i = jp + 1; i <= j; ++i) cut[i] = k;       // first bin above points jp + 1 .. j
        float fall = 0.f, rise = 0.f;
        if (j >= 0 && j <= nm) {
            const double d = 1.0 / fmax(pts[j + 1] - pts[j], 1e-9);
            if (j >= 1) fall = (float)fmax(0.0, fmin(1.0, (pts[j + 1] - f) * d));
            if (j < nm) rise = (float)fmax(0.0, fmin(1.0, (f - pts[j]) * d));
        }
        w1[k] = fall;
        w2[k] = rise;
    }
    __syncthreads();

    const int grp = threadIdx.x / kFeatThreads, tid = threadIdx.x - grp * kFeatThreads;
    unsigned char *gs = fsm + FL.group + grp * FL.group_bytes;
    const int fr = tid >> 7, ft = tid & 127;                // frame of the pair, thread in it
    const int XS = fpad(m) + 1;
    float2 *X0 = reinterpret_cast<float2 *>(gs + FL.X) + fr * XS, *X1 = X0 + 2 * XS;
    float *P = reinterpret_cast<float *>(gs + FL.P);
    float *accs = reinterpret_cast<float *>(gs + FL.acc);
    constexpr int kAcc = 2 * kFeatMaxMels / kFeatThreads;
    const long long items = (long long)S * A.batch, stride = (long long)gridDim.x * A.groups;
    for (long long item = blockIdx.x + (long long)gridDim.x * grp; item < items; item += stride) {
        const int b = (int)(item / S), s = (int)(item - (long long)b * S);
        const int f0 = (int)(((long long)s * F) / S);
        int f1 = (int)(((long long)(s + 1) * F) / S);
        f1 = min(max(f1, f0 + 1), F);
        const float *x = A.audio + (long long)b * T;
        float acc[kAcc];
#pragma unroll
        for (int q = 0; q < kAcc; ++q) acc[q] = 0.f;
        for (int f = f0; f < f1; f += 2) {
            const int ff = f + fr;
            const bool live = ff < f1;
            // pass 1 from global memory: windowed sample pairs (2 j, 2 j + 1), no twiddles
            auto sample = [&](int i) {
                int t = ff * hop + i - m;
                if (t < 0) t = -t;
                if (t >= T) t = 2 * (T - 1) - t;
                return win[i] * x[t];
            };
            const int base = ff * hop - m;
            const bool inside = base >= 0 && base + n <= T;
            for (int j = ft; j < m / 4; j += 128) {
                float2 v[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int i = 2 * (j + r * (m / 4));
                    v[r] = make_float2(0.f, 0.f);
                    if (live)
                        v[r] = inside ? make_float2(win[i] * x[base + i], win[i + 1] * x[base + i + 1])
                                      : make_float2(sample(i), sample(i + 1));
                }
                fft4(v);
#pragma unroll
                for (int r = 0; r < 4; ++r) X0[fpad(4 * j + r)] = v[r];
            }
            group_bar(grp);
            float2 *src = X0, *dst = X1;
            int ns = 4, lg = 2;
            for (; lg + 2 <= A.log2m; lg += 2, ns *= 4) {
                const int step = n / (4 * ns);                 // twiddle stride of W_{4 ns}
                for (int j = ft; j < m / 4; j += 128) {
                    const int k = j & (ns - 1);
                    float2 v[4];
                    v[0] = src[fpad(j)];
#pragma unroll
                    for (int r = 1; r < 4; ++r) v[r] = cmul(src[fpad(j + r * (m / 4))], tw[r * k * step]);
                    fft4(v);
                    const int o = (j - k) * 4 + k;
#pragma unroll
                    for (int r = 0; r < 4; ++r) dst[fpad(o + r * ns)] = v[r];
                }
                group_bar(grp);
                float2 *t = src;
                src = dst;
                dst = t;
            }
            if (lg < A.log2m) {
                for (int j = ft; j < m / 2; j += 128) {
                    const float2 a = src[fpad(j)], c = cmul(src[fpad(j + m / 2)], tw[2 * j]);
                    dst[fpad(j)] = make_float2(a.x + c.x, a.y + c.y);
                    dst[fpad(j + m / 2)] = make_float2(a.x - c.x, a.y - c.y);
                }
                group_bar(grp);
                src = dst;
            }
            // split: X[k] = E + W_n^k O with E, O the spectra of the even and odd samples
            for (int k = ft; k <= m; k += 128) {
                const float2 z = src[fpad(k & (m - 1))], y = src[fpad((m - k) & (m - 1))];
                const float2 E = make_float2(0.5f * (z.x + y.x), 0.5f * (z.y - y.y));
                const float2 O = make_float2(0.5f * (z.y + y.y), 0.5f * (y.x - z.x));
                const float2 wo = cmul(O, tw[k]);
                const float re = E.x + wo.x, im = E.y + wo.y;
                P[fr * (m + 1) + k] = re * re + im * im;
            }
            group_bar(grp);
#pragma unroll
            for (int q = 0; q < kAcc; ++q) {
                const int i = tid + q * kFeatThreads;          // (frame, filter)
                if (i >= 2 * nm) break;
                const int pf = i >= nm ? 1 : 0, mel = i - pf * nm;
                if (f + pf >= f1) continue;
                const float *Pf = P + pf * (m + 1);
                const int k0 = cut[mel], k1 = cut[mel + 1], k2 = cut[mel + 2];
                float v = 0.f;
#pragma unroll 4
                for (int k = k0; k < k1; ++k) v = fmaf(w2[k], Pf[k], v);
#pragma unroll 4
                for (int k = k1; k < k2; ++k) v = fmaf(w1[k], Pf[k], v);
                acc[q] += logf(v + 1e-6f);
            }
            group_bar(grp);     // the buffers are free for the next pair
        }
#pragma unroll
        for (int q = 0; q < kAcc; ++q) {
            const int i = tid + q * kFeatThreads;
            if (i < 2 * nm) accs[i] = acc[q];
        }
        group_bar(grp);
        for (int mel = tid; mel < nm; mel += kFeatThreads)
            A.out[((long long)b * nm + mel) * S + s] = (accs[mel] + accs[nm + mel]) / (float)(f1 - f0);
        group_bar(grp);
    }
}

}  // namespace

}  // namespace mdx

extern "C" int mdx_logmel(const float *audio, int batch, int T, double fs, int n_fft, int hop,
                          int n_mels, double fmin, double fmax, int segments, float *out,
                          void *stream) {
    using namespace mdx;
    if (!audio || !out) return set_last_error(MDX_ERR_ARG, "audio and out are required");
    if (batch < 1 || segments < 1) return set_last_error(MDX_ERR_ARG, "batch and segments must be >= 1");
    if (n_fft < 16 || n_fft > 2048 || (n_fft & (n_fft - 1)) != 0)
        return set_last_error(MDX_ERR_ARG, "n_fft must be a power of two in [16, 2048]");
    int log2n = 0;
    while ((1 << log2n) < n_fft) ++log2n;
    if (hop < 1) return set_last_error(MDX_ERR_ARG, "hop must be >= 1");
    if (T <= n_fft / 2) return set_last_error(MDX_ERR_ARG, "T must exceed n_fft / 2 (reflection padding)");
    if (1 + T / hop < segments) return set_last_error(MDX_ERR_ARG, "fewer frames than segments");
    if (n_mels < 1 || n_mels > kFeatMaxMels)
        return set_last_error(MDX_ERR_ARG, "n_mels must be in [1, 512]");
    if (!(fs > 0.0) || !(fmin >= 0.0) || !(fmax > fmin) || fmax > fs / 2.0)
        return set_last_error(MDX_ERR_ARG, "need 0 <= fmin < fmax <= fs / 2");
    // persistent CTAs, one per SM of the current device, with as many groups as its
    // shared memory holds; never more CTAs than (segment, signal) items
    int dev = 0, sms = 1, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaFuncSetAttribute(logmel_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin) !=
            cudaSuccess)
        return set_last_error(MDX_ERR_CUDA, "no usable current device");
    const FeatLayout L = feat_layout(n_fft, n_mels);
    const int groups = std::min<int>(kFeatGroups, (int)(((size_t)optin - L.group) / L.group_bytes));
    const long long items = (long long)segments * batch;
    LogmelArgs A{audio, batch, T, n_fft, log2n - 1, hop, n_mels, segments, groups, fs, fmin, fmax, out};
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    logmel_kernel<<<(unsigned)std::min<long long>(items, sms), groups * kFeatThreads,
                    L.group + groups * L.group_bytes, s>>>(A);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_last_error(MDX_ERR_CUDA, cudaGetErrorString(e));
    return MDX_OK;
}
