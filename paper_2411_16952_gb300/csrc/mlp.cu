// mlp.cu - the learned proposal: a 4 -> 64 -> 64 -> 64 MLP that maps a
// parameter point (K, E0, beta', C3/C2) to per-mode log-variance corrections
// c_k of the paper's proposal, sigma_k'^2 = sigma_k^2 e^{c_k}.
//
// The proposal stays a projected centred Gaussian, so its density against the
// uniform measure keeps the closed form of Eqs. (33)-(38):
//   g(xh) = prod_k w'_k Q^-K,  w'_k = 1/sigma_k'^2,  Q = sum_k w'_k s_k,
// and the accept test of Eq. (40) stays exact with K ln Q and a recomputed
// envelope M.  Training minimises, per point and over accepted samples i
// (draws from f), the tempered negative log-likelihood
//   J_tau = tau log mean_i exp((z_i + ell_i)/tau),  ell_i = K ln Q_i - sum ln w'_k,
// with z_i = -beta H_i (tau = inf: the plain mean, i.e. KL(f || g) + const);
// small tau weights the draws with the largest f/g, which set the acceptance.
//
// Parameters are held as FP32 masters (Adam) and used as BF16 copies in every
// forward and backward pass; all sums accumulate in FP32.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "../../include/tkdv.h"
#include "tkdv_internal.h"

namespace tkdv {
namespace mlpk {

constexpr int H = 64, KO = 64, NIN = 4;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + H * NIN, OFF_W2 = OFF_B1 + H, OFF_B2 = OFF_W2 + H * H,
              OFF_W3 = OFF_B2 + H, OFF_B3 = OFF_W3 + KO * H, NPARAM = OFF_B3 + KO;
static_assert(NPARAM == TKDV_MLP_NPARAM, "parameter count");

__device__ __forceinline__ float bf(const __nv_bfloat16 *w, int i) { return __bfloat162float(w[i]); }

// A row of 64 BF16 weights as eight 16-byte loads, and its FMA chain onto a.
struct WRow {
    uint4 v[8];
    __device__ __forceinline__ void load(const __nv_bfloat16 *w) {
#pragma unroll
        for (int i = 0; i < 8; ++i)  // (volatile: not moved behind the first barrier)
            asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(v[i].x), "=r"(v[i].y), "=r"(v[i].z), "=r"(v[i].w)
                         : "l"(reinterpret_cast<const uint4 *>(w) + i));
    }
    __device__ __forceinline__ float chain(float a, const float *x) const {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t u[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                a = fmaf(__uint_as_float(u[e] << 16), x[8 * i + 2 * e], a);
                a = fmaf(__uint_as_float(u[e] & 0xFFFF0000u), x[8 * i + 2 * e + 1], a);
            }
        }
        return a;
    }
};
static_assert(OFF_W2 % 8 == 0 && OFF_W3 % 8 == 0, "the weight rows start on 16-byte boundaries");

// Forward pass of P points, one CTA of 64 threads per point.  Both 64 x 64
// layers' rows are on their way before the first tanh (with loads of single
// weights as they were needed the pass took 8 us).  With Ks not null also what
// the loss needs: gauge-fixed c (mean zero over k < K), w'_k = w_k e^{-c_k},
// and the constant sum_k ln w'_k.
__global__ void __launch_bounds__(64) k_forward(const __nv_bfloat16 *__restrict__ w, const float *__restrict__ feats,
                                                float *h1, float *h2, float *out, const int *__restrict__ Ks,
                                                const float *__restrict__ wpaper, float *wprime, float *sumlogw) {
    const int p = blockIdx.x, j = threadIdx.x;
    __shared__ float sf[NIN], s1[H], s2[H], red[64];
    WRow w2, w3;
    w2.load(w + OFF_W2 + j * H);
    w3.load(w + OFF_W3 + j * H);
    if (j < NIN) sf[j] = feats[p * NIN + j];
    __syncthreads();
    float a = bf(w, OFF_B1 + j);
#pragma unroll
    for (int i = 0; i < NIN; ++i) a = fmaf(bf(w, OFF_W1 + j * NIN + i), sf[i], a);
    const float t1 = tanhf(a);
    s1[j] = t1;
    h1[p * H + j] = t1;
    __syncthreads();
    const float t2 = tanhf(w2.chain(bf(w, OFF_B2 + j), s1));
    s2[j] = t2;
    h2[p * H + j] = t2;
    __syncthreads();
    a = w3.chain(bf(w, OFF_B3 + j), s2);
    out[p * KO + j] = a;
    if (!Ks) return;
    const int k = j, K = Ks[p];
    const float o = k < K ? a : 0.f;
    red[k] = o;
    __syncthreads();
    for (int s = 32; s > 0; s >>= 1) {
        if (k < s) red[k] += red[k + s];
        __syncthreads();
    }
    const float mean = red[0] / (float)K;
    __syncthreads();
    const float c = o - mean;
    const float wv = k < K ? wpaper[p * KO + k] * expf(-c) : 0.f;
    wprime[p * KO + k] = wv;
    red[k] = k < K ? logf(wv) : 0.f;
    __syncthreads();
    for (int s = 32; s > 0; s >>= 1) {
        if (k < s) red[k] += red[k + s];
        __syncthreads();
    }
    if (k == 0) sumlogw[p] = red[0];
}

// Loss and its gradient at the output: grid (nblk, P), 256 threads.  A warp
// streams 32 rows (of `stride` floats: s_1..s_K, zero padded) at a time, LPR
// lanes to a row with four columns each, so that its loads are runs of whole
// rows; the lanes' shares of Q = sum w'_k s_k meet in a transposed reduction
// that leaves every lane with one row's Q.  Each lane then has a_i = (z_i +
// ell_i)/tau of one row (tau <= 0 means tau = inf, a_i = 0), the warp keeps a
// common running maximum m, and the weighted sums V_k = sum e^{a_i - m} s_ik/Q_i
// (four columns per lane), S = sum e^{a_i - m} and L = sum e^{a_i - m} ell_i.
// The last block of a point merges the blocks' [m, S, L, V_1..V_64].
//
// What bounds it: HBM, the rows are read once.  8 x 2^20 rows of 32 modes (1.1
// GB) take 163 us here, the rate of a plain copy; with a row per thread (loads 128 bytes apart, 64
// registers of w' and V per thread and a serial merge kernel) it was 289 + 24.
template <int LPR>
__global__ void __launch_bounds__(256) k_loss(const float *__restrict__ s, const float *__restrict__ z,
                                              const unsigned long long *__restrict__ row0,
                                              const unsigned long long *__restrict__ nrows, const int *__restrict__ Ks,
                                              const float *__restrict__ wprime, const float *__restrict__ sumlogw,
                                              int stride, float tau, float *partial, uint32_t *done, float *dout,
                                              float *loss) {
    constexpr int RPW = 32 / LPR;  // rows of one load
    constexpr int PSTR = KO + 3;
    __shared__ float s_v[8][KO], s_m[8], s_s[8], s_l[8];
    __shared__ bool s_last;
    const int p = blockIdx.y, K = Ks[p], t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int c = lane % LPR, sub = lane / LPR;
    const unsigned long long n = nrows[p];
    const float slw = sumlogw[p];
    const bool col = 4 * c < stride;
    float4 w = make_float4(0.f, 0.f, 0.f, 0.f), V = w;
    if (col) w = *reinterpret_cast<const float4 *>(wprime + p * KO + 4 * c);  // zero from K on
    const float *sp = s + row0[p] * (unsigned long long)stride + 4 * c, *zp = z + row0[p];
    float m = -INFINITY, S = 0.f, L = 0.f;
    for (unsigned long long r0 = 32ull * (blockIdx.x * 8ull + (unsigned)warp); r0 < n; r0 += 256ull * gridDim.x) {
        float4 v[LPR];
        float q[LPR];
#pragma unroll
        for (int b = 0; b < LPR; ++b) {
            const unsigned long long r = r0 + (unsigned)(b * RPW + sub);
            v[b] = col && r < n ? __ldcs(reinterpret_cast<const float4 *>(sp + r * (unsigned)stride))
                                : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const unsigned long long mine = r0 + (unsigned)(c * RPW + sub);
        const bool valid = mine < n;
        const float zi = valid ? __ldcs(zp + mine) : 0.f;
#pragma unroll
        for (int b = 0; b < LPR; ++b)
            q[b] = fmaf(w.w, v[b].w, fmaf(w.z, v[b].z, fmaf(w.y, v[b].y, w.x * v[b].x)));
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int e = 0; e < o; ++e) {
                const float send = up ? q[e] : q[e + o], keep = up ? q[e + o] : q[e];
                q[e] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
        const float Q = valid ? q[0] : 1.f;
        const float ell = (float)K * logf(Q) - slw;
        const float a = !valid ? -INFINITY : tau > 0.f ? (zi + ell) / tau : 0.f;
        if (__any_sync(0xffffffffu, a > m)) {
            float mn = fmaxf(m, a);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            const float scale = expf(m - mn);  // 0 on the first rows
            S *= scale;
            L *= scale;
            V = make_float4(V.x * scale, V.y * scale, V.z * scale, V.w * scale);
            m = mn;
        }
        const float e = valid ? expf(a - m) : 0.f;
        S += e;
        L = fmaf(e, ell, L);
        const float eq = e / Q;
        float4 d = make_float4(0.f, 0.f, 0.f, 0.f);  // of these rows alone: V's chain stays short
#pragma unroll
        for (int b = 0; b < LPR; ++b) {
            const float f = __shfl_sync(0xffffffffu, eq, sub * LPR + b);
            d.x = fmaf(f, v[b].x, d.x);
            d.y = fmaf(f, v[b].y, d.y);
            d.z = fmaf(f, v[b].z, d.z);
            d.w = fmaf(f, v[b].w, d.w);
        }
        V = make_float4(V.x + d.x, V.y + d.y, V.z + d.z, V.w + d.w);
    }
    // the block's sums: m is common to a warp, so the warps' sums scale to the
    // block's maximum
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        S += __shfl_xor_sync(0xffffffffu, S, o);
        L += __shfl_xor_sync(0xffffffffu, L, o);
        if (o >= LPR) {
            V.x += __shfl_xor_sync(0xffffffffu, V.x, o);
            V.y += __shfl_xor_sync(0xffffffffu, V.y, o);
            V.z += __shfl_xor_sync(0xffffffffu, V.z, o);
            V.w += __shfl_xor_sync(0xffffffffu, V.w, o);
        }
    }
    for (int e = t; e < 8 * KO; e += 256) (&s_v[0][0])[e] = 0.f;
    if (lane == 0) {
        s_m[warp] = m;
        s_s[warp] = S;
        s_l[warp] = L;
    }
    __syncthreads();
    if (lane < LPR) *reinterpret_cast<float4 *>(&s_v[warp][4 * lane]) = V;
    __syncthreads();
    float M = -INFINITY;
    for (int e = 0; e < 8; ++e) M = fmaxf(M, s_m[e]);
    float *out = partial + ((size_t)p * gridDim.x + blockIdx.x) * PSTR;
    if (t < PSTR) {
        float x = 0.f;
        for (int e = 0; e < 8; ++e) {
            const float f = s_m[e] == -INFINITY ? 0.f : expf(s_m[e] - M);
            x = fmaf(f, t == 1 ? s_s[e] : t == 2 ? s_l[e] : t >= 3 ? s_v[e][t - 3] : 0.f, x);
        }
        out[t] = t == 0 ? M : x;
    }
    __threadfence();
    __syncthreads();
    if (t == 0) s_last = atomicAdd(&done[p], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    // the point's last block: loss J_p and dJ/dc_raw (through the gauge); four
    // groups of 64 threads take every fourth block each
    __threadfence();
    if (t == 0) done[p] = 0;  // for the next step
    const volatile float *pp = partial + (size_t)p * gridDim.x * PSTR;
    const int k = t & 63, g = t >> 6, nblk = gridDim.x;
    float Mb = -INFINITY;
    for (int b = t; b < nblk; b += 256) Mb = fmaxf(Mb, pp[b * PSTR]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) Mb = fmaxf(Mb, __shfl_xor_sync(0xffffffffu, Mb, o));
    __syncthreads();
    if (lane == 0) s_m[warp] = Mb;
    __syncthreads();
    M = -INFINITY;
    for (int e = 0; e < 8; ++e) M = fmaxf(M, s_m[e]);
    float Sg = 0.f, Lg = 0.f, Vg = 0.f;
    for (int b = g; b < nblk; b += 4) {
        const float mb = pp[b * PSTR];
        const float f = mb == -INFINITY ? 0.f : expf(mb - M);
        Sg = fmaf(f, pp[b * PSTR + 1], Sg);
        Lg = fmaf(f, pp[b * PSTR + 2], Lg);
        Vg = fmaf(f, pp[b * PSTR + 3 + k], Vg);
    }
    s_v[g][k] = Vg;
    if (k == 0) {
        s_s[g] = Sg;
        s_l[g] = Lg;
    }
    __syncthreads();
    float *red = s_v[4];
    if (t >= 64) return;
    const float St = (s_s[0] + s_s[1]) + (s_s[2] + s_s[3]), Lt = (s_l[0] + s_l[1]) + (s_l[2] + s_l[3]);
    const float Vt = (s_v[0][k] + s_v[1][k]) + (s_v[2][k] + s_v[3][k]);
    // dJ/dc_k = 1 - K w'_k V_k / S   (k < K); zero mean over k < K already
    const float gk = k < K ? 1.f - (float)K * wprime[p * KO + k] * Vt / St : 0.f;
    red[k] = gk;
    asm volatile("bar.sync 1, 64;" ::: "memory");
    for (int s2 = 32; s2 > 0; s2 >>= 1) {
        if (k < s2) red[k] += red[k + s2];
        asm volatile("bar.sync 1, 64;" ::: "memory");
    }
    const float mean = red[0] / (float)K;
    dout[p * KO + k] = k < K ? gk - mean : 0.f;
    if (k == 0) loss[p] = tau > 0.f ? (float)((double)tau * ((double)M + log((double)St / (double)n))) : Lt / St;
}

// Backward pass through the MLP for all points, and with update the Adam step
// on the FP32 masters: one thread per parameter.  Every block makes da2 and
// da1 of all points for itself (P x 64 x 64 x 2 FMAs from shared memory, less
// than a hand-over between kernels would take); the new BF16 copies go to
// another buffer than the weights that other blocks still read.  grad (NPARAM
// floats) receives the sum over points.  One block for everything, and a
// second kernel for Adam, took 23 + 4 us.
__global__ void __launch_bounds__(256) k_backward(const __nv_bfloat16 *__restrict__ w, const float *__restrict__ feats,
                                                  const float *__restrict__ h1, const float *__restrict__ h2,
                                                  const float *__restrict__ dout, int P, float *grad, int update,
                                                  float *master, float *m1, float *m2, __nv_bfloat16 *wb, float lr,
                                                  float b1, float b2, float eps, float c1, float c2) {
    extern __shared__ float s_da[];  // da2 [P][64], da1 [P][64]
    __shared__ __align__(16) __nv_bfloat16 s_w[2][KO * H];  // W3, W2
    const int t = threadIdx.x;
    for (int e = t; e < KO * H / 8; e += 256) {
        reinterpret_cast<uint4 *>(s_w[0])[e] = __ldg(reinterpret_cast<const uint4 *>(w + OFF_W3) + e);
        reinterpret_cast<uint4 *>(s_w[1])[e] = __ldg(reinterpret_cast<const uint4 *>(w + OFF_W2) + e);
    }
    float *da2 = s_da, *da1 = s_da + P * H;
    __syncthreads();
    // da2[p][i] = (sum_j dout[p][j] W3[j][i]) (1 - h2^2)
    for (int e = t; e < P * H; e += 256) {
        const int p = e / H, i = e % H;
        float a = 0.f;
#pragma unroll 16
        for (int j = 0; j < KO; ++j) a = fmaf(__ldg(dout + p * KO + j), bf(s_w[0], j * H + i), a);
        const float hv = h2[p * H + i];
        da2[e] = a * (1.f - hv * hv);
    }
    __syncthreads();
    for (int e = t; e < P * H; e += 256) {
        const int p = e / H, i = e % H;
        float a = 0.f;
#pragma unroll 16
        for (int j = 0; j < H; ++j) a = fmaf(da2[p * H + j], bf(s_w[1], j * H + i), a);
        const float hv = h1[p * H + i];
        da1[e] = a * (1.f - hv * hv);
    }
    __syncthreads();
    const int i = blockIdx.x * 256 + t;
    if (i >= NPARAM) return;
    // the parameter's gradient: sum over p of d[p][row] x[p][column], or of d[p][row] for a bias
    const float *d, *x = nullptr;
    int row, colx = 0, xs = H;
    if (i >= OFF_B3) {
        d = dout, row = i - OFF_B3;
    } else if (i >= OFF_W3) {
        d = dout, x = h2, row = (i - OFF_W3) / H, colx = (i - OFF_W3) % H;
    } else if (i >= OFF_B2) {
        d = da2, row = i - OFF_B2;
    } else if (i >= OFF_W2) {
        d = da2, x = h1, row = (i - OFF_W2) / H, colx = (i - OFF_W2) % H;
    } else if (i >= OFF_B1) {
        d = da1, row = i - OFF_B1;
    } else {
        d = da1, x = feats, row = i / NIN, colx = i % NIN, xs = NIN;
    }
    float g = 0.f;
    if (x)
        for (int p = 0; p < P; ++p) g = fmaf(d[p * H + row], x[p * xs + colx], g);
    else
        for (int p = 0; p < P; ++p) g += d[p * H + row];
    grad[i] = g;
    if (!update) return;
    const float a = b1 * m1[i] + (1.f - b1) * g;
    const float b = b2 * m2[i] + (1.f - b2) * g * g;
    m1[i] = a;
    m2[i] = b;
    const float v = master[i] - lr * (a / c1) / (sqrtf(b / c2) + eps);
    master[i] = v;
    wb[i] = __float2bfloat16_rn(v);
}
static_assert(KO == H, "the rows of dout and da have the same length");

// BF16 copies of new masters; Adam starts again.
__global__ void k_set_params(const float *master, __nv_bfloat16 *wb, float *m1, float *m2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NPARAM) return;
    wb[i] = __float2bfloat16_rn(master[i]);
    m1[i] = 0.f;
    m2[i] = 0.f;
}

// Training rows from the sampler's accepted records: s_k = xh_k^2 + xh_{K+k}^2
// and z = -beta H = -beta'/(E0 K^2) (H2 - r H3), scattered per point.
__global__ void k_records_to_rows(const unsigned char *__restrict__ ring, unsigned long long nrec, int rec_bytes,
                                  int K, int stride, const unsigned long long *__restrict__ row0,
                                  const unsigned long long *__restrict__ cap, unsigned long long *fill,
                                  const float *__restrict__ zcoef /* per point: beta'/(E0 K^2), r */, float *s,
                                  float *z) {
    const unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nrec) return;
    const unsigned char *rec = ring + i * (unsigned long long)rec_bytes;
    const uint32_t p = *reinterpret_cast<const uint32_t *>(rec + 8);
    const unsigned long long slot = atomicAdd(&fill[p], 1ull);
    if (slot >= cap[p]) return;
    const float *f = reinterpret_cast<const float *>(rec + 16);
    const float *xh = f + 4;
    float *row = s + (row0[p] + slot) * (unsigned long long)stride;
    for (int k = 0; k < stride; ++k) row[k] = k < K ? xh[k] * xh[k] + xh[K + k] * xh[K + k] : 0.f;
    z[row0[p] + slot] = -zcoef[2 * p] * (f[0] - zcoef[2 * p + 1] * f[1]);
}

}  // namespace mlpk
}  // namespace tkdv

using namespace tkdv;
using namespace tkdv::mlpk;

struct tkdv_mlp {
    float *d_master = nullptr, *d_m1 = nullptr, *d_m2 = nullptr, *d_grad = nullptr;
    __nv_bfloat16 *d_wb[2] = {nullptr, nullptr};  // the copies in use, and the ones an update writes
    int cur = 0;
    float *h_lg = nullptr;  // pinned: losses of up to 64 points, then the gradient (laid out as d_loss | d_grad)
    // training set
    int P = 0, stride = 4, kmax = 4;
    std::vector<int> K;
    float *d_feats = nullptr, *d_wpaper = nullptr, *d_s = nullptr, *d_z = nullptr;
    unsigned long long *d_row0 = nullptr, *d_nrows = nullptr;
    std::vector<unsigned long long> nrows;
    int *d_K = nullptr;
    // work buffers
    float *d_h1 = nullptr, *d_h2 = nullptr, *d_out = nullptr, *d_wprime = nullptr, *d_slw = nullptr,
          *d_partial = nullptr, *d_dout = nullptr, *d_loss = nullptr;
    uint32_t *d_done = nullptr;  // finished blocks of each point's loss
    int nblk = 0;
    int step = 0;
    std::string err;
};

namespace {

int mfail(tkdv_mlp *m, int code, const std::string &msg) {
    if (m) m->err = msg;
    return code;
}

#define MCK(call)                                                                      \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess)                                                         \
            return mfail(m, e_ == cudaErrorMemoryAllocation ? TKDV_ERR_OOM : TKDV_ERR_CUDA, \
                         std::string(#call) + ": " + cudaGetErrorString(e_));          \
    } while (0)

void free_set(tkdv_mlp *m) {
    for (void *p : {(void *)m->d_feats, (void *)m->d_wpaper, (void *)m->d_s, (void *)m->d_z, (void *)m->d_row0,
                    (void *)m->d_nrows, (void *)m->d_K, (void *)m->d_h1, (void *)m->d_h2, (void *)m->d_out,
                    (void *)m->d_wprime, (void *)m->d_slw, (void *)m->d_partial, (void *)m->d_dout,
                    (void *)m->d_done})
        if (p) cudaFree(p);
    m->d_feats = m->d_wpaper = m->d_s = m->d_z = nullptr;
    m->d_row0 = m->d_nrows = nullptr;
    m->d_K = nullptr;
    m->d_h1 = m->d_h2 = m->d_out = m->d_wprime = m->d_slw = m->d_partial = m->d_dout = nullptr;
    m->d_done = nullptr;
    m->P = 0;
}

const void *loss_kernel(int kmax) {
    if (kmax <= 16) return (const void *)k_loss<4>;
    if (kmax <= 32) return (const void *)k_loss<8>;
    return (const void *)k_loss<16>;
}

// Work buffers for P points.
int alloc_work(tkdv_mlp *m, int P) {
    // the blocks of all points together fill the device once
    int dev = 0, sms = 0, per_sm = 0;
    MCK(cudaGetDevice(&dev));
    MCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    MCK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, loss_kernel(m->kmax), 256, 0));
    m->nblk = std::max(1, sms * std::max(1, per_sm) / P);
    MCK(cudaMalloc(&m->d_h1, sizeof(float) * P * H));
    MCK(cudaMalloc(&m->d_h2, sizeof(float) * P * H));
    MCK(cudaMalloc(&m->d_out, sizeof(float) * P * KO));
    MCK(cudaMalloc(&m->d_wprime, sizeof(float) * P * KO));
    MCK(cudaMalloc(&m->d_slw, sizeof(float) * P));
    MCK(cudaMalloc(&m->d_partial, sizeof(float) * P * m->nblk * (KO + 3)));
    MCK(cudaMalloc(&m->d_dout, sizeof(float) * P * KO));
    MCK(cudaMalloc(&m->d_done, sizeof(uint32_t) * P));
    MCK(cudaMemset(m->d_done, 0, sizeof(uint32_t) * P));
    return TKDV_OK;
}

}  // namespace

extern "C" {

int tkdv_mlp_features(int K, double beta_p, double E0, double r, double *out4) {
    if (!out4 || K < 1 || K > 64 || !(E0 > 0)) return TKDV_ERR_INVALID_ARG;
    const double lam = beta_p * r;
    out4[0] = std::log(std::max(beta_p, 1e-3)) / std::log(100.0);
    out4[1] = std::log(E0);
    out4[2] = std::log1p(std::max(lam, 0.0) / 100.0) / std::log(100.0);
    out4[3] = K / 64.0;
    return TKDV_OK;
}

int tkdv_mlp_create(uint64_t seed, tkdv_mlp **out) {
    if (!out) return TKDV_ERR_INVALID_ARG;
    *out = nullptr;
    tkdv_mlp *m = new tkdv_mlp();
    std::vector<float> w(NPARAM, 0.f);
    std::mt19937_64 gen(seed);
    std::normal_distribution<float> nd(0.f, 1.f);
    for (int i = 0; i < H * NIN; ++i) w[OFF_W1 + i] = 0.3f * nd(gen);
    for (int i = 0; i < H * H; ++i) w[OFF_W2 + i] = 0.15f * nd(gen);  // W3, biases: zero (c = 0 at start)
    auto bail = [&](int rc) {
        tkdv_mlp_destroy(m);
        return rc;
    };
    int rc;
    if ((rc = cudaMalloc(&m->d_master, 4 * NPARAM)) || (rc = cudaMalloc(&m->d_m1, 4 * NPARAM)) ||
        (rc = cudaMalloc(&m->d_m2, 4 * NPARAM)) || (rc = cudaMalloc(&m->d_loss, 4 * (TKDV_MAX_POINTS + NPARAM))) ||
        (rc = cudaMalloc(&m->d_wb[0], 2 * NPARAM)) || (rc = cudaMalloc(&m->d_wb[1], 2 * NPARAM)) ||
        (rc = cudaMallocHost(&m->h_lg, 4 * (TKDV_MAX_POINTS + NPARAM))))
        return bail(rc == cudaErrorMemoryAllocation ? TKDV_ERR_OOM : TKDV_ERR_CUDA);
    m->d_grad = m->d_loss + TKDV_MAX_POINTS;
    cudaError_t e = cudaMemcpy(m->d_master, w.data(), 4 * NPARAM, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_set_params<<<(NPARAM + 255) / 256, 256>>>(m->d_master, m->d_wb[0], m->d_m1, m->d_m2);
        e = cudaDeviceSynchronize();
    }
    if (e != cudaSuccess) return bail(TKDV_ERR_CUDA);
    *out = m;
    return TKDV_OK;
}

void tkdv_mlp_destroy(tkdv_mlp *m) {
    if (!m) return;
    free_set(m);
    for (void *p : {(void *)m->d_master, (void *)m->d_m1, (void *)m->d_m2, (void *)m->d_loss, (void *)m->d_wb[0],
                    (void *)m->d_wb[1]})
        if (p) cudaFree(p);
    if (m->h_lg) cudaFreeHost(m->h_lg);
    delete m;
}

const char *tkdv_mlp_last_error(const tkdv_mlp *m) { return m ? m->err.c_str() : ""; }

int tkdv_mlp_get_params(tkdv_mlp *m, float *master, float *bf16_values) {
    if (!m) return TKDV_ERR_INVALID_ARG;
    if (master) MCK(cudaMemcpy(master, m->d_master, 4 * NPARAM, cudaMemcpyDeviceToHost));
    if (bf16_values) {
        std::vector<uint16_t> b(NPARAM);
        MCK(cudaMemcpy(b.data(), m->d_wb[m->cur], 2 * NPARAM, cudaMemcpyDeviceToHost));
        for (int i = 0; i < NPARAM; ++i) {
            const uint32_t u = (uint32_t)b[i] << 16;
            std::memcpy(&bf16_values[i], &u, 4);
        }
    }
    return TKDV_OK;
}

int tkdv_mlp_set_params(tkdv_mlp *m, const float *master) {
    if (!m || !master) return TKDV_ERR_INVALID_ARG;
    MCK(cudaMemcpy(m->d_master, master, 4 * NPARAM, cudaMemcpyHostToDevice));
    m->step = 0;
    k_set_params<<<(NPARAM + 255) / 256, 256>>>(m->d_master, m->d_wb[m->cur], m->d_m1, m->d_m2);
    MCK(cudaDeviceSynchronize());
    return TKDV_OK;
}

int tkdv_mlp_infer(tkdv_mlp *m, int P, const double *feats, const int *K, double *c_out) {
    if (!m || P < 1 || P > TKDV_MAX_POINTS || !feats || !K || !c_out) return TKDV_ERR_INVALID_ARG;
    for (int p = 0; p < P; ++p)
        if (K[p] < 1 || K[p] > 64) return mfail(m, TKDV_ERR_INVALID_ARG, "K must be in 1..64");
    std::vector<float> f(P * NIN);
    for (int i = 0; i < P * NIN; ++i) f[i] = (float)feats[i];
    float *d_f = nullptr, *d_h = nullptr, *d_o = nullptr;
    MCK(cudaMalloc(&d_f, 4 * P * NIN));
    cudaError_t e = cudaMalloc(&d_h, 4 * P * H * 2);
    if (e == cudaSuccess) e = cudaMalloc(&d_o, 4 * P * KO);
    if (e == cudaSuccess) e = cudaMemcpy(d_f, f.data(), 4 * P * NIN, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_forward<<<P, 64>>>(m->d_wb[m->cur], d_f, d_h, d_h + P * H, d_o, nullptr, nullptr, nullptr, nullptr);
        e = cudaDeviceSynchronize();
    }
    std::vector<float> o(P * KO);
    if (e == cudaSuccess) e = cudaMemcpy(o.data(), d_o, 4 * P * KO, cudaMemcpyDeviceToHost);
    cudaFree(d_f);
    cudaFree(d_h);
    cudaFree(d_o);
    if (e != cudaSuccess) return mfail(m, TKDV_ERR_CUDA, std::string("infer: ") + cudaGetErrorString(e));
    for (int p = 0; p < P; ++p) {
        double mean = 0;
        for (int k = 0; k < K[p]; ++k) mean += o[p * KO + k];
        mean /= K[p];
        for (int k = 0; k < KO; ++k) c_out[p * KO + k] = k < K[p] ? (double)o[p * KO + k] - mean : 0.0;
    }
    return TKDV_OK;
}

int tkdv_mlp_set_data(tkdv_mlp *m, int P, const int *K, const double *feats, const double *w_paper,
                      const uint64_t *counts, const float *s_rows, const float *z) {
    if (!m || P < 1 || P > TKDV_MAX_POINTS || !K || !feats || !w_paper || !counts || !s_rows)
        return TKDV_ERR_INVALID_ARG;
    free_set(m);
    m->P = P;
    m->K.assign(K, K + P);
    m->kmax = 1;
    for (int p = 0; p < P; ++p) {
        if (K[p] < 1 || K[p] > 64) return mfail(m, TKDV_ERR_INVALID_ARG, "K must be in 1..64");
        m->kmax = std::max(m->kmax, K[p]);
    }
    m->stride = (m->kmax + 3) / 4 * 4;
    m->nrows.assign(counts, counts + P);
    std::vector<unsigned long long> row0(P, 0);
    unsigned long long tot = 0;
    for (int p = 0; p < P; ++p) {
        row0[p] = tot;
        tot += counts[p];
        if (counts[p] == 0) return mfail(m, TKDV_ERR_INVALID_ARG, "every point needs samples");
    }
    std::vector<float> f(P * NIN), wp(P * KO, 0.f);
    for (int i = 0; i < P * NIN; ++i) f[i] = (float)feats[i];
    for (int p = 0; p < P; ++p)
        for (int k = 0; k < K[p]; ++k) wp[p * KO + k] = (float)w_paper[p * KO + k];
    std::vector<float> zz(tot, 0.f);
    if (z) std::memcpy(zz.data(), z, 4 * tot);
    MCK(cudaMalloc(&m->d_feats, 4 * P * NIN));
    MCK(cudaMalloc(&m->d_wpaper, 4 * P * KO));
    MCK(cudaMalloc(&m->d_s, 4 * tot * m->stride));
    MCK(cudaMalloc(&m->d_z, 4 * tot));
    MCK(cudaMalloc(&m->d_row0, 8 * P));
    MCK(cudaMalloc(&m->d_nrows, 8 * P));
    MCK(cudaMalloc(&m->d_K, 4 * P));
    MCK(cudaMemcpy(m->d_feats, f.data(), 4 * P * NIN, cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(m->d_wpaper, wp.data(), 4 * P * KO, cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(m->d_s, s_rows, 4 * tot * m->stride, cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(m->d_z, zz.data(), 4 * tot, cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(m->d_row0, row0.data(), 8 * P, cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(m->d_nrows, m->nrows.data(), 8 * P, cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(m->d_K, m->K.data(), 4 * P, cudaMemcpyHostToDevice));
    return alloc_work(m, P);
}

int tkdv_mlp_set_data_records(tkdv_mlp *m, int P, const int *K, const double *feats, const double *w_paper,
                              const double *zcoef, const void *records_dev, uint64_t n_records, int K_records,
                              uint64_t max_per_point) {
    if (!m || P < 1 || P > TKDV_MAX_POINTS || !K || !feats || !w_paper || !zcoef || (!records_dev && n_records) ||
        max_per_point == 0 || K_records < 1 || K_records > 64)
        return TKDV_ERR_INVALID_ARG;
    for (int p = 0; p < P; ++p)
        if (K[p] != K_records) return mfail(m, TKDV_ERR_INVALID_ARG, "all points must have the records' K");
    free_set(m);
    m->P = P;
    m->K.assign(K, K + P);
    m->kmax = K_records;
    m->stride = (K_records + 3) / 4 * 4;
    std::vector<unsigned long long> row0(P), cap(P, max_per_point);
    for (int p = 0; p < P; ++p) row0[p] = (unsigned long long)p * max_per_point;
    const unsigned long long tot = (unsigned long long)P * max_per_point;
    std::vector<float> f(P * NIN), wp(P * KO, 0.f), zc(2 * P);
    for (int i = 0; i < P * NIN; ++i) f[i] = (float)feats[i];
    for (int p = 0; p < P; ++p) {
        for (int k = 0; k < K[p]; ++k) wp[p * KO + k] = (float)w_paper[p * KO + k];
        zc[2 * p] = (float)zcoef[2 * p];
        zc[2 * p + 1] = (float)zcoef[2 * p + 1];
    }
    unsigned long long *d_cap = nullptr, *d_fill = nullptr;
    float *d_zc = nullptr;
    MCK(cudaMalloc(&m->d_feats, 4 * P * NIN));
    MCK(cudaMalloc(&m->d_wpaper, 4 * P * KO));
    MCK(cudaMalloc(&m->d_s, 4 * tot * m->stride));
    MCK(cudaMalloc(&m->d_z, 4 * tot));
    MCK(cudaMalloc(&m->d_row0, 8 * P));
    MCK(cudaMalloc(&m->d_nrows, 8 * P));
    MCK(cudaMalloc(&m->d_K, 4 * P));
    MCK(cudaMalloc(&d_cap, 8 * P));
    MCK(cudaMalloc(&d_fill, 8 * P));
    MCK(cudaMalloc(&d_zc, 4 * 2 * P));
    MCK(cudaMemcpy(m->d_feats, f.data(), 4 * P * NIN, cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(m->d_wpaper, wp.data(), 4 * P * KO, cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(m->d_row0, row0.data(), 8 * P, cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(m->d_K, m->K.data(), 4 * P, cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(d_cap, cap.data(), 8 * P, cudaMemcpyHostToDevice));
    MCK(cudaMemcpy(d_zc, zc.data(), 8 * P, cudaMemcpyHostToDevice));
    MCK(cudaMemset(d_fill, 0, 8 * P));
    if (n_records) {
        const int rb = (int)record_bytes(K_records);
        k_records_to_rows<<<(unsigned)((n_records + 255) / 256), 256>>>((const unsigned char *)records_dev, n_records,
                                                                        rb, K_records, m->stride, m->d_row0, d_cap,
                                                                        d_fill, d_zc, m->d_s, m->d_z);
    }
    std::vector<unsigned long long> fill(P);
    MCK(cudaMemcpy(fill.data(), d_fill, 8 * P, cudaMemcpyDeviceToHost));
    cudaFree(d_cap);
    cudaFree(d_fill);
    cudaFree(d_zc);
    m->nrows.resize(P);
    for (int p = 0; p < P; ++p) {
        m->nrows[p] = std::min<unsigned long long>(fill[p], max_per_point);
        if (m->nrows[p] == 0) return mfail(m, TKDV_ERR_INVALID_ARG, "a point has no accepted records");
    }
    MCK(cudaMemcpy(m->d_nrows, m->nrows.data(), 8 * P, cudaMemcpyHostToDevice));
    return alloc_work(m, P);
}

int tkdv_mlp_rows(tkdv_mlp *m, uint64_t *counts) {
    if (!m || !counts) return TKDV_ERR_INVALID_ARG;
    for (int p = 0; p < m->P; ++p) counts[p] = m->nrows[p];
    return TKDV_OK;
}

int tkdv_mlp_step(tkdv_mlp *m, float lr, float tau, int update, double *loss, float *grad_out) {
    if (!m || m->P < 1) return TKDV_ERR_INVALID_ARG;
    if (!m->d_done) return mfail(m, TKDV_ERR_INVALID_ARG, "the training set was refused");  // (allocated last)
    const int P = m->P;
    const __nv_bfloat16 *wb = m->d_wb[m->cur];
    MCK(launch_kernel(k_forward, P, 64, 0, 0, wb, m->d_feats, m->d_h1, m->d_h2, m->d_out, m->d_K, m->d_wpaper, m->d_wprime,
                      m->d_slw));
    {
        const float *s = m->d_s, *z = m->d_z, *wpr = m->d_wprime, *slw = m->d_slw;
        const unsigned long long *r0 = m->d_row0, *nr = m->d_nrows;
        const int *Kd = m->d_K;
        int stride = m->stride;
        float t = tau, *part = m->d_partial, *dout = m->d_dout, *dl = m->d_loss;
        uint32_t *done = m->d_done;
        void *args[] = {&s, &z, &r0, &nr, &Kd, &wpr, &slw, &stride, &t, &part, &done, &dout, &dl};
        MCK(cudaLaunchKernel(loss_kernel(m->kmax), dim3(m->nblk, P), dim3(256), args, 0, 0));
    }
    float c1 = 1.f, c2 = 1.f;
    const float b1 = 0.9f, b2 = 0.999f;
    if (update) {
        c1 = 1.f - std::pow(b1, (float)(m->step + 1));
        c2 = 1.f - std::pow(b2, (float)(m->step + 1));
    }
    MCK(launch_kernel(k_backward, (NPARAM + 255) / 256, 256, sizeof(float) * 2 * P * H, 0, wb, m->d_feats, m->d_h1, m->d_h2,
                      m->d_dout, P, m->d_grad, update ? 1 : 0, m->d_master, m->d_m1, m->d_m2, m->d_wb[m->cur ^ 1], lr, b1,
                      b2, 1e-8f, c1, c2));
    if (update) {  // the masters, their copies and the step count go together
        m->step += 1;
        m->cur ^= 1;
    }
    // losses and gradient in one copy
    if (loss || grad_out)
        MCK(cudaMemcpyAsync(m->h_lg, m->d_loss, 4 * (size_t)(grad_out ? TKDV_MAX_POINTS + NPARAM : P),
                            cudaMemcpyDeviceToHost, 0));
    MCK(cudaDeviceSynchronize());
    if (loss) {
        double t = 0;
        for (int p = 0; p < P; ++p) t += m->h_lg[p];
        *loss = t;
    }
    if (grad_out) std::memcpy(grad_out, m->h_lg + TKDV_MAX_POINTS, 4 * NPARAM);
    return TKDV_OK;
}

}  // extern "C"
