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
// What bounds it: an FP64 instruction of a warp holds its scheduler for 64
// cycles, and an iteration is a serial chain of about 300 of them at 64 modes
// (K triad products per lane pair, 12 inner products of the recursion).  All
// points and starts run at the same time, one warp each (616 warps on the 608
// schedulers for eight points at 64 modes), so the search of a handle takes
// about as long as its slowest start: 0.8 ms for eight points at 64 modes
// (25 evaluations a start on average), 6 ms for 32 points at 32 modes over two
// decades of beta', 1.9 ms for eight at 128 modes, where tkdv_log_M takes 107,
// 17 and 830 ms for each point on one host core.  A bisection step of eight
// 64-mode candidates went from 854 to 8.0 ms, a batch of 32 points at 32 modes
// from 541 to 14.1 ms, sampling included.
#include <cuda_runtime.h>
#include <math.h>

#include "sampler_impl.cuh"

namespace tkdv {
namespace {

constexpr int kHist = 6;      // remembered steps (12 took as many evaluations)
constexpr int kEnvWarps = 4;  // warps of a CTA, one per scheduler
constexpr int kEnvMaxIter = 3000, kEnvMaxHalvings = 60;

__device__ __forceinline__ double esum(double v) {
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

// F(y) and its gradient; xs: K doubles of the warp's shared memory; scale: the
// size of F's terms, whose last bits are the noise of F.
template <int VPL>
__device__ double env_eval(const EnvPoint *P, int K, const Lane<VPL> &L, double *xs, const double *y, double *g,
                           double &scale) {
    double nn = 0.0;
#pragma unroll
    for (int v = 0; v < VPL; ++v) nn = fma(y[v], y[v], nn);
    const double in = 1.0 / sqrt(esum(nn));
    double x[VPL], A[VPL], C[VPL];
    __syncwarp();
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
        x[v] = y[v] * in;
        if (L.on[v]) xs[L.i[v]] = x[v];
        A[v] = C[v] = 0.0;
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
        double s = 0.0, first = 0.0;
        int n = j0, k = 1;
        for (int t = 0; t < a0 + a1; ++t) {
            if (t == a0) {
                first = s;
                s = 0.0;
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
        s = first = 0.0;
        n = j0;
        k = 0;
        for (int t = 0; t < c0 + c1; ++t) {
            if (t == c0) {
                first = s;
                s = 0.0;
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
    double S = 0.0, Q = 0.0, T = 0.0, w[VPL], m2[VPL];
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
        const int n = L.i[v] + 1;
        w[v] = L.on[v] ? P->w[n - 1] : 0.0;
        m2[v] = (double)n * (double)n;
        A[v] *= 2.0;
        if ((n & 1) == 0) A[v] = fma(xs[n / 2 - 1], xs[n / 2 - 1], A[v]);
        if (L.on[v]) {
            const double xx = x[v] * x[v];
            S = fma(m2[v], xx, S);
            Q = fma(w[v], xx, Q);
            T = fma(x[v], A[v], T);
        }
    }
    S = esum(S);
    T = esum(T);
    double val = P->cS * S + P->cH * T, dot = 2.0 * P->cS * S + 3.0 * P->cH * T, wq = 0.0;
    scale = 1.0 + fabs(P->cS * S) + fabs(P->cH * T);
    if (P->cQ != 0.0) {
        Q = esum(Q);
        const double tQ = P->cQ * log(Q);
        val += tQ;
        scale += fabs(tQ);
        dot += 2.0 * P->cQ;  // g . x: S, T and ln Q are homogeneous (degrees 2, 3, and 2 inside the log)
        wq = 2.0 * P->cQ / Q;
    }
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
        const double gx = 2.0 * P->cS * m2[v] * x[v] + P->cH * (A[v] + 2.0 * C[v]) + wq * w[v] * x[v];
        g[v] = L.on[v] ? (gx - dot * x[v]) * in : 0.0;
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

template <int VPL>
__global__ void __launch_bounds__(32 * kEnvWarps) k_envelope(const EnvPoint *pts, int P, int K, int nstarts,
                                                             unsigned long long *best) {
    extern __shared__ double s_env[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int task = blockIdx.x * kEnvWarps + warp;
    if (task >= P * nstarts) return;  // whole warps leave
    const int p = task / nstarts;
    const EnvPoint *pt = pts + p;
    // the warp's shared memory: the evaluated state, and each lane's own
    // elements of the remembered steps S and gradient changes Y
    double *xs = s_env + (size_t)warp * (32 * VPL * (1 + 2 * kHist));
    double *hs = xs + 32 * VPL + lane;
    const Lane<VPL> L(lane, K);
    auto hS = [&](int slot, int v) -> double & { return hs[((2 * slot) * VPL + v) * 32]; };
    auto hY = [&](int slot, int v) -> double & { return hs[((2 * slot + 1) * VPL + v) * 32]; };
    auto dot = [&](const double *a, const double *b) {
        double s = 0.0;
#pragma unroll
        for (int v = 0; v < VPL; ++v) s = fma(a[v], b[v], s);
        return esum(s);
    };
    double y[VPL], g[VPL], yn[VPL], gn[VPL], d[VPL], rho[kHist], al[kHist];
    env_start<VPL>(task % nstarts, K, L, y);
    {
        const double in = 1.0 / sqrt(dot(y, y));
#pragma unroll
        for (int v = 0; v < VPL; ++v) y[v] *= in;
    }
    double scale;
    double f = env_eval<VPL>(pt, K, L, xs, y, g, scale);
    int hist = 0, head = 0, stall = 0, small = 0;  // slot of age a (0 the newest): head - 1 - a mod kHist
#pragma unroll 1
    for (int it = 0; it < kEnvMaxIter; ++it) {
        const double gg = dot(g, g);
        if (gg < 1e-26) break;
        // two-loop recursion for the ascent direction
#pragma unroll
        for (int v = 0; v < VPL; ++v) d[v] = g[v];
        double yy = 0.0, rnew = 0.0;
#pragma unroll
        for (int a = 0; a < kHist; ++a) {
            if (a < hist) {
                const int slot = (head - 1 - a + 2 * kHist) % kHist;
                double sv[VPL], yv[VPL], q2 = 0.0;
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
        const double gam = hist ? 1.0 / (rnew * yy) : 0.1 / sqrt(gg);
#pragma unroll
        for (int v = 0; v < VPL; ++v) d[v] *= gam;
#pragma unroll
        for (int a = kHist - 1; a >= 0; --a) {
            if (a < hist) {
                const int slot = (head - 1 - a + 2 * kHist) % kHist;
                double yv[VPL];
#pragma unroll
                for (int v = 0; v < VPL; ++v) yv[v] = hY(slot, v);
                const double b = al[a] - rho[a] * dot(yv, d);
#pragma unroll
                for (int v = 0; v < VPL; ++v) d[v] = fma(b, hS(slot, v), d[v]);
            }
        }
        double slope = dot(d, g);
        if (!(slope > 0.0)) {  // not an ascent direction: restart from the gradient
            hist = 0;
            const double c = 0.1 / sqrt(gg);
#pragma unroll
            for (int v = 0; v < VPL; ++v) d[v] = c * g[v];
            slope = 0.1 * sqrt(gg);
        }
        // the step promises less than the noise of F, twice: at the top.
        // (Going on until the gains vanish in the last bits took up to 413
        // evaluations instead of 55 at 64 modes, for the same 13 digits.)
        if (slope <= 1e-14 * scale) {
            if (++small >= 2) break;
        } else {
            small = 0;
        }
        double t = 1.0, fn = 0.0;
        bool ok = false;
#pragma unroll 1
        for (int ls = 0; ls < kEnvMaxHalvings; ++ls) {
#pragma unroll
            for (int v = 0; v < VPL; ++v) yn[v] = fma(t, d[v], y[v]);
            fn = env_eval<VPL>(pt, K, L, xs, yn, gn, scale);
            if (fn >= f + 1e-4 * t * slope) {
                ok = true;
                break;
            }
            t *= 0.5;
            if (t * slope < 1e-16 * scale) break;  // below the noise of F (halving on: 310 evaluations, not 48)
        }
        if (!ok) break;
        double sy = 0.0, ny = 0.0;
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            sy = fma(yn[v] - y[v], g[v] - gn[v], sy);
            ny = fma(yn[v], yn[v], ny);
        }
        sy = esum(sy);
        ny = esum(ny);
        if (sy > 1e-300) {
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                hS(head, v) = yn[v] - y[v];
                hY(head, v) = g[v] - gn[v];
            }
#pragma unroll
            for (int a = kHist - 1; a > 0; --a) rho[a] = rho[a - 1];  // rho by age
            rho[0] = 1.0 / sy;
            head = (head + 1) % kHist;
            hist = min(hist + 1, kHist);
        }
        const double gain = fn - f;
        f = fn;
        double sc = 1.0;
        if (ny > 4.0) {  // keep |y| near 1 (F does not depend on it)
            sc = sqrt(ny);
            hist = 0;
        }
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            y[v] = yn[v] / sc;
            g[v] = gn[v] * sc;
        }
        if (gain <= 1e-16 * (1.0 + fabs(f))) {
            if (++stall >= 8) break;
        } else {
            stall = 0;
        }
    }
    if (lane == 0 && f == f) atomicMax(&best[p], dkey(f));
}

template <int VPL>
cudaError_t launch(const EnvPoint *pts, int P, int K, unsigned long long *best, cudaStream_t st) {
    const int tasks = P * (K + 13);
    const size_t smem = sizeof(double) * kEnvWarps * 32 * VPL * (1 + 2 * kHist);
    cudaError_t e = cudaFuncSetAttribute(k_envelope<VPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_envelope<VPL><<<(tasks + kEnvWarps - 1) / kEnvWarps, 32 * kEnvWarps, smem, st>>>(pts, P, K, K + 13, best);
    return cudaGetLastError();
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
