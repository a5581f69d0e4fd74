// envelope.cu - the rejection constant M = sup f/g (Eq. 45) of all points of a
// handle, found on the device: one warp per (point, start).
//
// log f/g = cS S + cH T + cQ ln Q depends on the phases of the modes only
// through T, and |Re(v_k v_l conj v_{k+l})| <= |v_k||v_l||v_{k+l}|, so given the
// amplitudes |v_k| the largest cH T is |cH| times T of the real state with
// those amplitudes (T is odd).  The supremum over the sphere of 2K dimensions
// is therefore attained at real amplitudes, K dimensions, with cH replaced by
// |cH|: a quarter of the products per evaluation.  The search is L-BFGS ascent
// of F(y) = log f/g (y/|y|) in FP64 from the starts of tkdv_log_M
// (precompute.cpp, which searches the whole sphere on the host): the Dirichlet
// kernel, four tapered ones, every single mode with a nudge, and eight random
// amplitude vectors; the largest maximum wins.
//
// What bounds it: latency.  An iteration is a serial chain of about 300
// dependent instructions at 64 modes (K triad products per lane pair, 12 inner
// products of the recursion), and an FP64 instruction of a warp holds its
// scheduler for 64 cycles where an FP32 one takes 4.  So every start climbs in
// FP32 first, to within FP32's noise of a maximum, and FP64 goes on from there.
// All points and starts run at the same time, one warp each (616 warps on the
// 608 schedulers for eight points at 64 modes), so the search of a handle takes
// about as long as its slowest start: 0.4 ms for eight points at 64 modes, 1.7
// ms for 32 points at 32 modes over two decades of beta', 1.0 ms for eight at
// 128 modes (in FP64 throughout 0.8, 6.4 and 1.9 ms), where tkdv_log_M takes
// 107, 17 and 830 ms for each point on one host core.  A bisection step of
// eight 64-mode candidates went from 840 to 7.4 ms, a batch of 32 points at 32
// modes from 532 to 12.2 ms, sampling included.
#include <cuda_runtime.h>
#include <math.h>

#include "sampler_impl.cuh"

namespace tkdv {
namespace {

constexpr int kHist = 6;      // remembered steps (12 took as many evaluations)
constexpr int kEnvWarps = 4;  // warps of a CTA, one per scheduler
constexpr int kEnvMaxIter = 3000, kEnvMaxHalvings = 60;

template <typename R>
__device__ __forceinline__ R esum(R v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;  // the same bits in every lane
}

// Order-preserving map double -> uint64 (for atomicMax on signed values); 0 is
// below every value's key.
__device__ __forceinline__ unsigned long long dkey(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// Element v of a lane: modes in pairs (p + 1, K - p), p = lane + 32 q, v = 2q
// and 2q + 1, so that the sums of a pair together have the same length in
// every lane; with one element per lane (K <= 32) mode lane + 1.
template <int VPL>
struct Lane {
    int i[VPL];    // mode - 1
    bool on[VPL];  // the lane holds an element here
    __device__ Lane(int lane, int K) {
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            if (VPL == 1) {
                i[v] = lane;
                on[v] = lane < K;
            } else {
                const int p = lane + 32 * (v >> 1), m = K - 1 - p;
                i[v] = (v & 1) ? m : p;
                on[v] = (v & 1) ? m > p : m >= p;
            }
            if (!on[v]) i[v] = 0;
        }
    }
};

// F(y) and its gradient; xs: K values of the warp's shared memory; scale: the
// size of F's terms, whose last bits are the noise of F.
template <int VPL, typename R>
__device__ R env_eval(const EnvPoint *P, int K, const Lane<VPL> &L, R *xs, const R *y, R *g, R &scale) {
    const R cS = (R)P->cS, cH = (R)P->cH, cQ = (R)P->cQ;
    R nn = 0;
#pragma unroll
    for (int v = 0; v < VPL; ++v) nn = fma(y[v], y[v], nn);
    const R in = (R)1 / sqrt(esum(nn));
    R x[VPL], A[VPL], C[VPL];
    __syncwarp();
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
        x[v] = y[v] * in;
        if (L.on[v]) xs[L.i[v]] = x[v];
        A[v] = C[v] = 0;
    }
    __syncwarp();
    // A_n = sum_{k<n} x_k x_{n-k}, folded;  C_j = sum_{n>j} x_n x_{n-j}
#pragma unroll
    for (int v = 0; v < VPL; v += 2) {
        // the two elements of a pair as one loop (a switch of sums on the way)
        const bool two = VPL > 1;
        const int j0 = L.i[v] + 1, j1 = two ? L.i[v + (VPL > 1)] + 1 : 0;
        const bool on0 = L.on[v], on1 = two && L.on[v + (VPL > 1)];
        const int a0 = on0 ? (j0 - 1) / 2 : 0, a1 = on1 ? (j1 - 1) / 2 : 0;
        R s = 0, first = 0;
        int n = j0, k = 1;
        for (int t = 0; t < a0 + a1; ++t) {
            if (t == a0) {
                first = s;
                s = 0;
                n = j1;
                k = 1;
            }
            s = fma(xs[k - 1], xs[n - k - 1], s);
            ++k;
        }
        if (a1 > 0) {
            A[v] = first;
            A[v + (VPL > 1)] = s;
        } else {
            A[v] = s;
        }
        const int c0 = on0 ? K - j0 : 0, c1 = on1 ? K - j1 : 0;
        s = first = 0;
        n = j0;
        k = 0;
        for (int t = 0; t < c0 + c1; ++t) {
            if (t == c0) {
                first = s;
                s = 0;
                n = j1;
                k = 0;
            }
            s = fma(xs[n + k], xs[k], s);
            ++k;
        }
        if (c1 > 0) {
            C[v] = first;
            C[v + (VPL > 1)] = s;
        } else {
            C[v] = s;
        }
    }
    R S = 0, Q = 0, T = 0, w[VPL], m2[VPL];
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
        const int n = L.i[v] + 1;
        w[v] = L.on[v] ? (R)P->w[n - 1] : (R)0;
        m2[v] = (R)n * (R)n;
        A[v] *= (R)2;
        if ((n & 1) == 0) A[v] = fma(xs[n / 2 - 1], xs[n / 2 - 1], A[v]);
        if (L.on[v]) {
            const R xx = x[v] * x[v];
            S = fma(m2[v], xx, S);
            Q = fma(w[v], xx, Q);
            T = fma(x[v], A[v], T);
        }
    }
    S = esum(S);
    T = esum(T);
    R val = cS * S + cH * T, dot = (R)2 * cS * S + (R)3 * cH * T, wq = 0;
    scale = (R)1 + fabs(cS * S) + fabs(cH * T);
    if (cQ != (R)0) {
        Q = esum(Q);
        const R tQ = cQ * log(Q);
        val += tQ;
        scale += fabs(tQ);
        dot += (R)2 * cQ;  // g . x: S, T and ln Q are homogeneous (degrees 2, 3, and 2 inside the log)
        wq = (R)2 * cQ / Q;
    }
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
        const R gx = (R)2 * cS * m2[v] * x[v] + cH * (A[v] + (R)2 * C[v]) + wq * w[v] * x[v];
        g[v] = L.on[v] ? (gx - dot * x[v]) * in : (R)0;
    }
    return val;
}

// Start s of n = K + 13: see the head of the file.
template <int VPL>
__device__ void env_start(int s, int K, const Lane<VPL> &L, double *y) {
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
        const int i = L.i[v];
        const uint4 r = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)s, 0u, 0u), 0x7D0C5EEDu, 0u);
        double a;
        if (s == 0) {
            a = 1.0;
        } else if (s <= 4) {
            const double gam = s == 1 ? 0.5 : s == 2 ? 2.0 : s == 3 ? 8.0 : 32.0;
            a = exp(-gam * (double)((i + 1) * (i + 1)) / (double)(K * K));
        } else if (s < 5 + K) {
            a = i == s - 5 ? 1.0 : 1e-3 * u01d(r.x);
        } else {
            a = -log(u01d(r.x));
        }
        y[v] = L.on[v] ? a : 0.0;
    }
}

// L-BFGS ascent of F from y, which receives the point reached; returns F
// there.  tol: noise of F relative to its terms.  xs: the warp's shared memory.
template <int VPL, typename R>
__device__ R env_ascend(const EnvPoint *pt, int K, const Lane<VPL> &L, R *xs, R *y, R tol, int max_iter) {
    const int lane = threadIdx.x & 31;
    // after the evaluated state, each lane's own elements of the remembered
    // steps S and gradient changes Y
    R *hs = xs + 32 * VPL + lane;
    auto hS = [&](int slot, int v) -> R & { return hs[((2 * slot) * VPL + v) * 32]; };
    auto hY = [&](int slot, int v) -> R & { return hs[((2 * slot + 1) * VPL + v) * 32]; };
    auto dot = [&](const R *a, const R *b) {
        R s = 0;
#pragma unroll
        for (int v = 0; v < VPL; ++v) s = fma(a[v], b[v], s);
        return esum(s);
    };
    R g[VPL], yn[VPL], gn[VPL], d[VPL], rho[kHist], al[kHist];
    {
        const R in = (R)1 / sqrt(dot(y, y));
#pragma unroll
        for (int v = 0; v < VPL; ++v) y[v] *= in;
    }
    R scale;
    R f = env_eval<VPL, R>(pt, K, L, xs, y, g, scale);
    int hist = 0, head = 0, stall = 0, small = 0;  // slot of age a (0 the newest): head - 1 - a mod kHist
#pragma unroll 1
    for (int it = 0; it < max_iter; ++it) {
        const R gg = dot(g, g);
        if (gg < (R)1e-26) break;
        // two-loop recursion for the ascent direction
#pragma unroll
        for (int v = 0; v < VPL; ++v) d[v] = g[v];
        R yy = 0, rnew = 0;
#pragma unroll
        for (int a = 0; a < kHist; ++a) {
            if (a < hist) {
                const int slot = (head - 1 - a + 2 * kHist) % kHist;
                R sv[VPL], yv[VPL], q2 = 0;
#pragma unroll
                for (int v = 0; v < VPL; ++v) {
                    sv[v] = hS(slot, v);
                    yv[v] = hY(slot, v);
                }
                al[a] = rho[a] * dot(sv, d);
#pragma unroll
                for (int v = 0; v < VPL; ++v) {
                    d[v] = fma(-al[a], yv[v], d[v]);
                    q2 = fma(yv[v], yv[v], q2);
                }
                if (a == 0) {
                    yy = esum(q2);
                    rnew = rho[0];
                }
            }
        }
        const R gam = hist ? (R)1 / (rnew * yy) : (R)0.1 / sqrt(gg);
#pragma unroll
        for (int v = 0; v < VPL; ++v) d[v] *= gam;
#pragma unroll
        for (int a = kHist - 1; a >= 0; --a) {
            if (a < hist) {
                const int slot = (head - 1 - a + 2 * kHist) % kHist;
                R yv[VPL];
#pragma unroll
                for (int v = 0; v < VPL; ++v) yv[v] = hY(slot, v);
                const R b = al[a] - rho[a] * dot(yv, d);
#pragma unroll
                for (int v = 0; v < VPL; ++v) d[v] = fma(b, hS(slot, v), d[v]);
            }
        }
        R slope = dot(d, g);
        if (!(slope > (R)0)) {  // not an ascent direction: restart from the gradient
            hist = 0;
            const R c = (R)0.1 / sqrt(gg);
#pragma unroll
            for (int v = 0; v < VPL; ++v) d[v] = c * g[v];
            slope = (R)0.1 * sqrt(gg);
        }
        // the step promises less than the noise of F, twice: at the top.
        // (Going on until the gains vanish in the last bits took up to 413
        // evaluations instead of 55 at 64 modes, for the same 13 digits.)
        if (slope <= tol * scale) {
            if (++small >= 2) break;
        } else {
            small = 0;
        }
        R t = 1, fn = 0;
        bool ok = false;
#pragma unroll 1
        for (int ls = 0; ls < kEnvMaxHalvings; ++ls) {
#pragma unroll
            for (int v = 0; v < VPL; ++v) yn[v] = fma(t, d[v], y[v]);
            fn = env_eval<VPL, R>(pt, K, L, xs, yn, gn, scale);
            if (fn >= f + (R)1e-4 * t * slope) {
                ok = true;
                break;
            }
            t *= (R)0.5;
            if (t * slope < (R)0.01 * tol * scale) break;  // below the noise of F (halving on: 310 evaluations, not 48)
        }
        if (!ok) break;
        R sy = 0, ny = 0;
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            sy = fma(yn[v] - y[v], g[v] - gn[v], sy);
            ny = fma(yn[v], yn[v], ny);
        }
        sy = esum(sy);
        ny = esum(ny);
        if (sy > (sizeof(R) == 8 ? (R)1e-300 : (R)1e-30)) {
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                hS(head, v) = yn[v] - y[v];
                hY(head, v) = g[v] - gn[v];
            }
#pragma unroll
            for (int a = kHist - 1; a > 0; --a) rho[a] = rho[a - 1];  // rho by age
            rho[0] = (R)1 / sy;
            head = (head + 1) % kHist;
            hist = min(hist + 1, kHist);
        }
        const R gain = fn - f;
        f = fn;
        R sc = 1;
        if (ny > (R)4) {  // keep |y| near 1 (F does not depend on it)
            sc = sqrt(ny);
            hist = 0;
        }
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            y[v] = yn[v] / sc;
            g[v] = gn[v] * sc;
        }
        if (gain <= (R)0.01 * tol * ((R)1 + fabs(f))) {
            if (++stall >= 8) break;
        } else {
            stall = 0;
        }
    }
    return f;
}

template <int VPL>
__global__ void __launch_bounds__(32 * kEnvWarps) k_envelope(const EnvPoint *pts, int P, int K, int nstarts,
                                                             unsigned long long *best) {
    extern __shared__ double s_env[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int task = blockIdx.x * kEnvWarps + warp;
    if (task >= P * nstarts) return;  // whole warps leave
    const int p = task / nstarts;
    const EnvPoint *pt = pts + p;
    double *xs = s_env + (size_t)warp * (32 * VPL * (1 + 2 * kHist));
    const Lane<VPL> L(lane, K);
    double y[VPL];
    float yf[VPL];
    env_start<VPL>(task % nstarts, K, L, y);
#pragma unroll
    for (int v = 0; v < VPL; ++v) yf[v] = (float)y[v];
    // FP32 first: it brings every start, and the slow ones above all, to within
    // its noise of a maximum at a tenth of the cost; then FP64 from there (from
    // the start itself if FP32 overflowed)
    const float ff = env_ascend<VPL, float>(pt, K, L, reinterpret_cast<float *>(xs), yf, 3e-7f, kEnvMaxIter);
    bool fine = fabsf(ff) < INFINITY;
#pragma unroll
    for (int v = 0; v < VPL; ++v) fine = fine && fabsf(yf[v]) < INFINITY;
    if (__all_sync(0xffffffffu, fine)) {
#pragma unroll
        for (int v = 0; v < VPL; ++v) y[v] = L.on[v] ? (double)yf[v] : 0.0;
    }
    __syncwarp();
    const double f = env_ascend<VPL, double>(pt, K, L, xs, y, 1e-14, kEnvMaxIter);
    if (lane == 0 && f == f) atomicMax(&best[p], dkey(f));
}

template <int VPL>
cudaError_t launch(const EnvPoint *pts, int P, int K, unsigned long long *best, cudaStream_t st) {
    const int tasks = P * (K + 13);
    const size_t smem = sizeof(double) * kEnvWarps * 32 * VPL * (1 + 2 * kHist);
    cudaError_t e = cudaFuncSetAttribute(k_envelope<VPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_kernel(k_envelope<VPL>, (tasks + kEnvWarps - 1) / kEnvWarps, 32 * kEnvWarps, smem, st, pts, P, K, K + 13,
                         best);
}

}  // namespace

cudaError_t launch_envelope(const EnvPoint *pts, int P, int K, unsigned long long *best, cudaStream_t st) {
    if (K <= 32) return launch<1>(pts, P, K, best, st);
    if (K <= 64) return launch<2>(pts, P, K, best, st);
    return launch<4>(pts, P, K, best, st);
}

double envelope_value(unsigned long long key) {
    if (key == 0) return -INFINITY;
    const unsigned long long b = (key >> 63) ? key & 0x7FFFFFFFFFFFFFFFull : ~key;
    double v;
    memcpy(&v, &b, 8);
    return v;
}

}  // namespace tkdv
