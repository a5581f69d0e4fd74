// sampler_k128.cu - the rejection sampler for 65..128 modes (Sec. IV.B of
// Moore & Foerster, arXiv 2411.16952, at the K = 128 of Fig. 7): one warp per
// batch of four proposals, the batch's state in shared memory.
//
// At K = 128 one proposal holds 256 floats, too many for one thread's
// registers, and the double sum of Eq. (42) has 4096 distinct triads.  So a
// warp draws four proposals at once: lane L makes modes 2j, 2j+1 for the
// Philox blocks j = L and L + 32 of every proposal (the stream rule of the
// one-thread sampler, so both forms draw the same states), writes the scaled
// pairs (x_m, y_m) to shared memory and keeps its share of |x|^2, S|x|^2,
// Q|x|^2, u(0) and the smallest radius word, which warp reductions complete.
//
// H3 is the grid cubature of Eq. (2) by a fast transform in FP32, eight lanes
// per proposal.  With C(xi) = sum x_k cos k xi and S(xi) = sum y_k sin k xi the
// field at +-xi is proportional to C +- S, and a pair of points contributes
// 2 C (C^2 + 3 S^2).  2 (C + i S) = sum_k (x_k + y_k) e^{ik xi} + (x_k - y_k)
// e^{-ik xi} has real coefficients c_k, k = 1..128 and -1..-128, so on the
// N = 384 points xi_j = 2 pi (j + 1/2)/N the points j and N - 1 - j are
// conjugate and N/2 = 192 values suffice.  With k = k1 + 24 k2 and j = j2 + 16
// j1 (j2 even: one of each conjugate pair)
//   value_j = sum_{k1} e^{2 pi i k1 j1/24} [e^{i pi k1 (2 j2 + 1)/384}
//             sum_{k2} c_{k1 + 24 k2} e^{2 pi i k2 (j2 + 1/2)/16}];
// the inner sum over 16 real c, X_n and X_{n+8} joined to X_n + i X_{n+8}, is
// an 8-point transform of (X_n + i X_{n+8}) e^{2 pi i n/32}, whose results are
// j2 = 0, 2, .., 14.  A lane makes three of the 24 columns k1, twists and
// stores them, and takes one j2: 24 = 3 x 8 points without further twists
// (3 and 8 have no common factor), cubed and summed as they come.  N = 384 =
// 3 x 128 points do not integrate e^{+-i 384 xi}: the cube of mode 128 alone
// aliases, and its term (N/4) Re v_128^3, with the sign of the half-step
// offset, is added back.
//
// What bounds it: issue of the FP32 and integer pipes.  The transform is about
// 6,400 thread instructions per proposal; 8 x 8 tiles of the double sum of
// Eq. (42), the form before, took 26,000 (4608 packed products of 2 cycles
// each, their loads and the tiles' ends), of 33,300 in all; now 20,100 in all,
// issue 75 % busy (60 % before).  2 x 2^21 proposals at acceptance 0.28: 6.58 ms
// with the tiles, 3.90 ms with the transform, 3.43 ms with the draw loop rolled
// up, the shared Philox rounds, and the spectrum of accepted draws in
// registers (64-bit float conversions run on the FP64 pipe, 12 % busy with
// them).  The transform's error in H3 against FP64, with that of the draw, is
// 4.8e-7 of the root mean square (3.8e-7 with the tiles; nearly all of the
// difference to log f/(Mg), 1.2e-5, is the draw's and unchanged).  It serves the
// decision; H3 and log f/(Mg) of a kept record have the double sum (fold_T, 3.8e-7).
//
// Rounding: the 2-norm of the 192 values is off by at most 25 roundings
// (coefficients 1, three-level 8-point transforms 5 each, twists 3 each, the
// 3-point one 3), which moves T by 2 sqrt(K) of it, and the sum of the cubes
// adds chains of at most 13 terms: 75 2^-24 sqrt(K), against the 512 2^-24
// sqrt(K) of the decision guard of point_table.cpp, so the guard band and the
// FP64 pass (k_refine_warp) keep every accept decision exact.  The radius is
// rho_log, the full-precision logarithm, whose error is purely relative: the
// guard needs no per-draw radius terms and is about ten times narrower than
// it would be with the fast radius, so that about 0.15 % of the draws at
// K = 128 reach the FP64 pass.
//
// Shared memory of a warp: proposal q's state at float2 word q * kWS, mode m
// (from 0) at word m, modes K..127 zero; then its transform at q * kWB, value
// (l, k1) at word kWR l + k1.  The strides put the eight lanes of the two
// proposals of a half-warp on distinct banks in every access.
#include "sampler_impl.cuh"

namespace tkdv {
namespace {

constexpr int kWK = 128;  // modes of the layout
constexpr int kWQ = 4;    // proposals per warp batch, eight lanes each
constexpr int kWN = 384;  // grid points
constexpr int kWS = 136;  // float2 words of one proposal's state
constexpr int kWR = 25;   // float2 words of one row (24 columns) of the transform
constexpr int kWB = 8 * kWR;  // float2 words of one proposal's transform
constexpr int kWarpWords = kWQ * (kWS + kWB);  // float2 words of a warp's slab

struct cf {
    float x, y;
};
__device__ __forceinline__ cf operator+(cf a, cf b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ cf operator-(cf a, cf b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ cf cmul(cf a, float c, float s) {
    return {fmaf(a.x, c, -(a.y * s)), fmaf(a.x, s, a.y * c)};
}
__device__ __forceinline__ cf muli(cf a) { return {-a.y, a.x}; }

// z_k = sum_n z_n e^{2 pi i n k/8}, in place.
__device__ __forceinline__ void dft8(cf *z) {
    constexpr float r = 0.70710678118654752440f;
    const cf a0 = z[0] + z[4], a1 = z[0] - z[4], a2 = z[2] + z[6], a3 = muli(z[2] - z[6]);
    const cf b0 = z[1] + z[5], b1 = z[1] - z[5], b2 = z[3] + z[7], b3 = muli(z[3] - z[7]);
    const cf e0 = a0 + a2, e2 = a0 - a2, e1 = a1 + a3, e3 = a1 - a3;
    const cf o0 = b0 + b2, o2 = muli(b0 - b2), o1 = b1 + b3, o3 = b1 - b3;
    z[0] = e0 + o0;
    z[4] = e0 - o0;
    z[2] = e2 + o2;
    z[6] = e2 - o2;
    // e^{i pi/4} o1 = r (o1.x - o1.y, o1.x + o1.y);  e^{3 i pi/4} o3 = r (-o3.x - o3.y, o3.x - o3.y)
    const float u = o1.x - o1.y, v = o1.x + o1.y, p = o3.x + o3.y, q = o3.x - o3.y;
    z[1] = {fmaf(r, u, e1.x), fmaf(r, v, e1.y)};
    z[5] = {fmaf(-r, u, e1.x), fmaf(-r, v, e1.y)};
    z[3] = {fmaf(-r, p, e3.x), fmaf(r, q, e3.y)};
    z[7] = {fmaf(r, p, e3.x), fmaf(-r, q, e3.y)};
}

// Twist of value (l, k1): e^{2 pi i k1 (4 l + 1)/768}, at word 24 l + k1.
__device__ __forceinline__ float2 twist_entry(int t) {
    const int l = t / 24, k1 = t % 24;
    float sn, cs;
    sincospif((float)(k1 * (4 * l + 1)) / 384.f, &sn, &cs);
    return make_float2(cs, sn);
}

// Column k1 = 8 C + s of a proposal: its 16 coefficients c_{k1 + 24 k2} (k <=
// 128 positive, k >= 256 standing for k - 384 with the sign of the half step), the 8-point transform, the
// twists, and the results to the rows l = 0..7 of wt.
template <int C>
__device__ __forceinline__ void column(const float2 *sv, float2 *wt, const float2 *tw, int s) {
    const int k1 = 8 * C + s;
    auto pos = [&](int k2) {  // x + y of mode k1 + 24 k2
        const float2 v = sv[k1 + 24 * k2 - 1];
        return v.x + v.y;
    };
    auto neg = [&](int k2) {  // -(x - y) of mode 384 - k1 - 24 k2: e^{-384 i xi_j} = -1
        const float2 v = sv[kWN - k1 - 24 * k2 - 1];
        return v.y - v.x;
    };
    // e^{2 pi i n/32}, n = 1..7
    constexpr float c1 = 0.98078528040323044913f, s1 = 0.19509032201612826785f, c2 = 0.92387953251128675613f,
                    s2 = 0.38268343236508977173f, c3 = 0.83146961230254523708f, s3 = 0.55557023301960222474f,
                    c4 = 0.70710678118654752440f;
    cf z[8];
    z[0] = {C > 0 || s > 0 ? pos(0) : 0.f, 0.f};  // (k = 0 has no mode)
    const float x1 = pos(1);
    z[1] = {x1 * c1, x1 * s1};
    const float x2 = pos(2);
    if (C == 2) {
        z[2] = cmul({x2, neg(10)}, c2, s2);  // k = 240 + k1 >= 256
    } else {
        z[2] = {x2 * c2, x2 * s2};
    }
    z[3] = cmul({pos(3), neg(11)}, c3, s3);
    z[4] = cmul({pos(4), neg(12)}, c4, c4);
    // k = 120 + k1 <= 128: all of column block 0, the first of block 1
    const float x5 = C == 0 ? pos(5) : C == 1 && s == 0 ? pos(5) : 0.f;
    z[5] = cmul({x5, neg(13)}, s3, c3);
    const float x6 = neg(14), x7 = neg(15);
    z[6] = {-x6 * c2, x6 * s2};  // i x6 e^{2 pi i 6/32}
    z[7] = {-x7 * c1, x7 * s1};  // i x7 e^{2 pi i 7/32}
    dft8(z);
#pragma unroll
    for (int l = 0; l < 8; ++l) {
        const float2 t = tw[24 * l + k1];
        const cf v = cmul(z[l], t.x, t.y);
        wt[kWR * l + k1] = make_float2(v.x, v.y);
    }
}

// sum of C (C^2 + 3 S^2) over the 24 points of row l = s.
__device__ __forceinline__ float row_cubes(const float2 *wr) {
    constexpr float h = 0.86602540378443864676f;
    cf z[3][8];
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        const float2 v0 = wr[(3 * a) % 24], v1 = wr[(3 * a + 8) % 24], v2 = wr[(3 * a + 16) % 24];
        const cf sm = {v1.x + v2.x, v1.y + v2.y}, d = {v1.x - v2.x, v1.y - v2.y};
        z[0][a] = {v0.x + sm.x, v0.y + sm.y};
        const cf t = {fmaf(-0.5f, sm.x, v0.x), fmaf(-0.5f, sm.y, v0.y)};
        z[1][a] = {fmaf(-h, d.y, t.x), fmaf(h, d.x, t.y)};
        z[2][a] = {fmaf(h, d.y, t.x), fmaf(-h, d.x, t.y)};
    }
    float acc[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        dft8(z[b]);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float c2 = z[b][j].x * z[b][j].x, s2 = z[b][j].y * z[b][j].y;
            acc[b] = fmaf(z[b][j].x, fmaf(3.f, s2, c2), acc[b]);
        }
    }
    return (acc[0] + acc[1]) + acc[2];
}

// One batch of the fast path: the four proposals' draws, reductions and T.
// On return every lane holds the values of proposal ql = lane & 3.
struct WEval {
    float nrm2, Sraw, zz, u0raw, T;
    bool tail;  // a radius word in the lowest bucket of the uniform map
};

// The lane's two Philox blocks (lane and lane + 32): their heads for the index
// half `hi` they were made for.
struct WHeads {
    PhiloxHead h[2];
    uint32_t hi;
    __device__ __forceinline__ void make(uint32_t hi_, uint32_t pid, const uint32_t *rk, int lane) {
        hi = hi_;
        h[0] = philox_head((uint32_t)lane, hi, pid, rk);
        h[1] = philox_head((uint32_t)lane + 32u, hi, pid, rk);
    }
};

// idx(q): the index of the batch's proposal q, q in vmask.
template <bool UNIF, typename Idx>
__device__ __forceinline__ WEval warp_batch(float2 *sv, const float2 *s_tw, const float *sig, const float *act, int K,
                                            const Idx &idx, uint32_t vmask, WHeads &heads, uint32_t pid,
                                            const uint32_t *rk, int lane) {
    uint32_t tails = 0;
    // Steps 1-3: lane L makes the Philox blocks L and L + 32 of every proposal.
    // The radius is rho_log (purely relative error), so the outputs of
    // accepted draws need no second pass and the guard no per-draw terms.  The
    // loop stays rolled: with the four proposals written out the loop body
    // (about 3,000 instructions) missed the instruction cache 1.2 times an
    // issue.  Partial sums |x|^2, S|x|^2, Q|x|^2 and u(0)|x|/u0s go to the
    // words of the transform, [q][lane] in steps of 4, 136 apart.
    float *part = reinterpret_cast<float *>(sv + kWQ * kWS);
#pragma unroll 1
    for (int q = 0; q < kWQ; ++q) {
        float nrm2 = 0.f, Sraw = 0.f, zz = 0.f, u0raw = 0.f;
        if ((vmask >> q) & 1u) {
            const unsigned long long id = idx(q);
            if ((uint32_t)(id >> 32) != heads.hi) heads.make((uint32_t)(id >> 32), pid, rk, lane);
            const PhiloxTail tail((uint32_t)id, heads.hi, rk);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int j = lane + 32 * i;
                if (2 * j < K) {
                    const uint4 w = tail.block(heads.h[i]);
                    float xy[4];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int m = 2 * j + h;
                        const float s = UNIF ? act[m] : sig[m];
                        const float rho = rho_log(h ? w.z : w.x);
                        const float a = (-s * rho) * rsqrt_approx(rho);
                        float sn, cs;
                        sincos_approx(angle_f(h ? w.w : w.y), sn, cs);
                        const float xm = a * cs, ym = a * sn;
                        if (m < K && (h ? w.z : w.x) < kTailBucket) tails |= 1u << q;
                        xy[2 * h] = xm;
                        xy[2 * h + 1] = ym;
                        const float sk = (s * s) * rho;
                        nrm2 += sk;
                        Sraw = fmaf((float)((m + 1) * (m + 1)), sk, Sraw);
                        zz += s > 0.f ? rho : 0.f;
                        u0raw += xm;
                    }
                    *reinterpret_cast<float4 *>(sv + q * kWS + 2 * j) = make_float4(xy[0], xy[1], xy[2], xy[3]);
                }
            }
        }
        *reinterpret_cast<float4 *>(part + q * 136 + 4 * lane) = make_float4(nrm2, Sraw, zz, u0raw);
    }
    tails = __reduce_or_sync(0xffffffffu, tails);
    __syncwarp();
    // The 16 sums over the warp: lanes 2 e and 2 e + 1 take sum e = 4 stat + q,
    // the partial sums of the even and of the odd lanes, in the order of a
    // butterfly (lanes 16, 8, 4 and 2 apart, then the two halves).
    float tot;
    {
        const float *src = part + ((lane >> 1) & 3) * 136 + 4 * (lane & 1) + (lane >> 3);
        float t[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) t[e] = src[8 * e] + src[8 * (e + 8)];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
#pragma unroll
            for (int e = 0; e < o; ++e) t[e] += t[e + o];
        tot = t[0] + __shfl_xor_sync(0xffffffffu, t[0], 1);
    }
    __syncwarp();
    // Step 4: the transform, eight lanes per proposal.
    const int q = lane >> 3, s = lane & 7;
    const float2 *xq = sv + q * kWS;
    float2 *wt = sv + kWQ * kWS + q * kWB;
    column<0>(xq, wt, s_tw, s);
    column<1>(xq, wt, s_tw, s);
    column<2>(xq, wt, s_tw, s);
    __syncwarp();
    float cub = row_cubes(wt + kWR * s);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) cub += __shfl_xor_sync(0xffffffffu, cub, o);
    const int ql = lane & 3;
    WEval ev;
    ev.nrm2 = __shfl_sync(0xffffffffu, tot, 2 * ql);
    ev.Sraw = __shfl_sync(0xffffffffu, tot, 8 + 2 * ql);
    ev.zz = __shfl_sync(0xffffffffu, tot, 16 + 2 * ql);
    ev.u0raw = __shfl_sync(0xffffffffu, tot, 24 + 2 * ql);
    // values and coefficients are 2 (C + i S): sum U^3 = 2 cub/8, less the
    // alias -(N/4) Re v_128^3, and T |x|^3 = (4/(3N)) sum U^3
    const float2 e = sv[ql * kWS + kWK - 1];
    const float alias = e.x * fmaf(e.x, e.x, -3.f * (e.y * e.y));
    ev.T = fmaf(__shfl_sync(0xffffffffu, cub, 8 * ql), 1.f / (3.f * kWN), alias * (1.f / 3.f));
    ev.tail = (tails >> ql) & 1u;
    return ev;
}

// T |x|^3 of a proposal whose H3 and log f/(Mg) are written out, by the double sum of Eq. (42),
// folded: T = sum_{n=2}^{K} Re(conj(v_n) W_n), W_n = 2 sum_{k < n-k} v_k v_{n-k} +
// [n even] v_{n/2}^2, a row n per lane, its products summed eight at a time.  Off
// by 1.2e-7 of the root mean square of T, where the transform is off by 2.6e-7
// (the draw adds 3.6e-7): the decision's guard covers that, the output keeps the
// double sum.  Bound by shared-memory loads, two for a product: 1.5 ns for a kept
// record at 128 modes (2 x 2^21 proposals, 1.16e6 accepted: 3.27 ms with a ring of
// 16 records, 5.00 ms with all kept; 6.52 ms when the tiles served every draw).
__device__ __forceinline__ float fold_T(const float2 *v, int K, int lane) {
    float t = 0.f;
#pragma unroll 1
    for (int n = 2 + lane; n <= K; n += 32) {
        float A = 0.f, B = 0.f;
        int k0 = 1;
#pragma unroll 1
        for (; 2 * (k0 + 7) < n; k0 += 8) {
            float a = 0.f, b = 0.f;
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                const float4 p = *reinterpret_cast<const float4 *>(v + k0 - 1 + j);  // modes k0 + j, k0 + j + 1
                const float2 q = v[n - k0 - j - 1], r = v[n - k0 - j - 2];
                a = fmaf(p.x, q.x, a);
                a = fmaf(-p.y, q.y, a);
                b = fmaf(p.x, q.y, b);
                b = fmaf(p.y, q.x, b);
                a = fmaf(p.z, r.x, a);
                a = fmaf(-p.w, r.y, a);
                b = fmaf(p.z, r.y, b);
                b = fmaf(p.w, r.x, b);
            }
            A += a;
            B += b;
        }
        float a = 0.f, b = 0.f;
#pragma unroll
        for (int k = k0; k < k0 + 7; ++k) {
            if (2 * k < n) {
                const float2 p = v[k - 1], q = v[n - k - 1];
                a = fmaf(p.x, q.x, a);
                a = fmaf(-p.y, q.y, a);
                b = fmaf(p.x, q.y, b);
                b = fmaf(p.y, q.x, b);
            }
        }
        A += a;
        B += b;
        A *= 2.f;
        B *= 2.f;
        if ((n & 1) == 0) {
            const float2 h = v[n / 2 - 1];
            A = fmaf(h.x, h.x, A);
            A = fmaf(-h.y, h.y, A);
            B = fmaf(2.f * h.x, h.y, B);
        }
        const float2 vn = v[n - 1];
        t = fmaf(vn.x, A, t);
        t = fmaf(vn.y, B, t);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// Steps 5-6 for the lane's proposal (the formulas of eval_fast).
template <bool UNIF>
__device__ __forceinline__ Fast warp_eval(const WEval &ev, const Scal &c, uint32_t wacc) {
    Fast f;
    const float inv2 = rcp_rn(ev.nrm2);
    f.inv = rsqrt_approx(ev.nrm2);
    f.S = ev.Sraw * inv2;
    f.T = ev.T * (inv2 * f.inv);
    const float tS = c.cS * f.S;
    const float tH = c.cH * f.T;
    const float tQ = UNIF ? 0.f : c.cQ * logf(ev.zz * inv2);
    f.delta = ((tS + tH) + tQ) - c.logM;
    f.lnU = -0.5f * rho_fast(wacc);
    f.d = f.lnU - f.delta;
    // the warp form's guard has no per-draw radius terms (guard_e = guard_q = 0)
    f.guard = c.ga + c.gr * (fabsf(tS) + fabsf(tQ) + fabsf(tH) + fabsf(f.lnU) + fabsf(c.logM)) + c.gh;
    return f;
}

// Shared state common to the sampler and the replay kernel: the twists and the
// proposal variances; the warps' slabs are zeroed (modes above K stay zero).
struct WShared {
    float2 tw[kWB];
    float sig[kWK], act[kWK];
};

__device__ void wshared_init(WShared &sh, float2 *slabs, int nw, int tid, int nt) {
    for (int t = tid; t < 8 * 24; t += nt) sh.tw[t] = twist_entry(t);
    for (int e = tid; e < nw * kWarpWords; e += nt) slabs[e] = make_float2(0.f, 0.f);
}

// ---- FP64 pass of the warp form -------------------------------------------
// The same draw and formulas as eval64 (sampler_impl.cuh), spread over a warp:
// lane L makes the modes of Philox blocks L and L + 32 into the slab sx (FP64
// pairs, zero from K on), and the double sum of Eq. (42), folded,
//   T = sum_{n=2}^{K} Re(conj(v_n) W_n),
//   W_n = 2 sum_{k < n-k} v_k v_{n-k} + [n even] v_{n/2}^2,
// takes rows n and 131 - n as one loop of 64 pairs (n = 3..65): two such
// loops per lane, and row 2 on lane 31.  Rows above K read v_n = 0.  Every
// lane returns the proposal's values.
__device__ __forceinline__ double wsum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ void row_end(const double2 *sx, int n, double A, double B, double &t) {
    A *= 2.0;
    B *= 2.0;
    if ((n & 1) == 0) {
        const double2 h = sx[n / 2 - 1];
        A = fma(h.x, h.x, A);
        A = fma(-h.y, h.y, A);
        B = fma(2.0 * h.x, h.y, B);
    }
    const double2 vn = sx[n - 1];
    t = fma(vn.x, A, t);
    t = fma(vn.y, B, t);
}

// rows n1 < n2 with (n1 - 1)/2 + (n2 - 1)/2 = 64 folded pairs
__device__ __forceinline__ void fold_pair(const double2 *sx, int n1, int n2, double &t) {
    const int len1 = (n1 - 1) / 2;
    double A = 0.0, B = 0.0;
    int n = n1, k = 1;
    for (int i = 0; i < 64; ++i) {
        if (i == len1) {
            row_end(sx, n1, A, B, t);
            A = 0.0;
            B = 0.0;
            n = n2;
            k = 1;
        }
        const double2 a = sx[k - 1], b = sx[n - k - 1];
        A = fma(a.x, b.x, A);
        A = fma(-a.y, b.y, A);
        B = fma(a.x, b.y, B);
        B = fma(a.y, b.x, B);
        ++k;
    }
    row_end(sx, n2, A, B, t);
}

template <bool UNIF>
__device__ __noinline__ void eval64_warp(const PointConst *P, unsigned long long idx, uint32_t k0, uint32_t k1,
                                         double2 *sx, int lane, Out64 &o, double &inv_out) {
    const int K = P->K;
    const uint32_t lo = (uint32_t)idx, hi = (uint32_t)(idx >> 32), pid = P->point_id;
    double nrm2 = 0.0, Sraw = 0.0, zz = 0.0, u0raw = 0.0;
    __syncwarp();  // earlier readers of the slab are done
    for (int jj = 0; jj < 2; ++jj) {
        const int j = lane + 32 * jj;
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (2 * j < K) w = philox4x32_10(make_uint4((uint32_t)j, lo, hi, pid), k0, k1);
        for (int h = 0; h < 2; ++h) {
            const int m = 2 * j + h;
            double2 v = make_double2(0.0, 0.0);
            if (m < K) {
                const double u1 = u01d_ext(h ? w.z : w.x, 2u * (uint32_t)m, lo, hi, pid, k0, k1);
                const double u2 = u01d(h ? w.w : w.y);
                const double rho = -2.0 * log(u1);
                const double rad = sqrt(rho);
                double sn, cs;
                sincospi(2.0 * u2, &sn, &cs);
                const double sg = UNIF ? 1.0 : P->sigma_d[m];
                v.x = sg * rad * cs;
                v.y = sg * rad * sn;
                const double sk = v.x * v.x + v.y * v.y;
                nrm2 += sk;
                Sraw += (double)((m + 1) * (m + 1)) * sk;
                zz += rho;
                u0raw += v.x;
            }
            sx[m] = v;
        }
    }
    __syncwarp();
    double t = 0.0;
    fold_pair(sx, 3 + lane, 128 - lane, t);
    if (lane < 31)
        fold_pair(sx, 35 + lane, 96 - lane, t);
    else
        row_end(sx, 2, 0.0, 0.0, t);
    const double T = wsum_d(t);
    nrm2 = wsum_d(nrm2);
    Sraw = wsum_d(Sraw);
    zz = wsum_d(zz);
    u0raw = wsum_d(u0raw);
    const double inv = 1.0 / sqrt(nrm2);
    const double inv2 = inv * inv;
    o.S = Sraw * inv2;
    o.T = T * inv2 * inv;
    double delta = P->cS_d * o.S + P->cH_d * o.T;
    if (!UNIF) delta += P->cQ_d * log(zz * inv2);
    delta -= P->logM;
    const uint32_t wa = accept_word(lo, hi, pid, K, k0, k1);
    o.delta = delta;
    o.u = u01d_ext(wa, 4u * (uint32_t)((K + 1) / 2), lo, hi, pid, k0, k1);
    o.lnU = log(o.u);
    o.accept = o.lnU < delta;
    o.near = fabs(o.lnU - delta) < 1e-6;
    o.H2 = (float)((double)P->E0 * o.S);
    o.H3 = (float)((double)P->h3s * o.T);
    o.u0 = (float)((double)P->u0s * u0raw * inv);
    inv_out = inv;
}

// FP64 decision of the guard-band proposals, one warp per queued proposal.
template <bool UNIF>
__global__ void __launch_bounds__(128) k_refine_warp(DevBufs B, uint32_t k0, uint32_t k1) {
    __shared__ double2 s_x[4][kWK];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double2 *sx = s_x[warp];
    const uint32_t n = min(*(volatile uint32_t *)&B.counters[1], B.refine_cap);
    for (uint32_t i = blockIdx.x * 4u + (uint32_t)warp; i < n; i += gridDim.x * 4u) {
        const RefineItem it = B.refine[i];
        const PointConst *P = B.pts + it.point;
        StatBlock *st = B.stats + it.point;
        Out64 o;
        double inv;
        eval64_warp<UNIF>(P, it.idx, k0, k1, sx, lane, o, inv);
        if (lane == 0) {
            atomicAdd(&st->n_refined, 1ull);
            atomicMax(&st->maxd_key, (unsigned long long)fkey((float)o.delta));
            if (o.near) atomicAdd(&st->n_near, 1ull);
            if (o.delta > 0.0) atomicAdd(&st->n_viol, 1ull);
        }
        if (!o.accept) continue;  // the same in every lane
        const int K = P->K;
        unsigned long long slot = 0;
        if (lane == 0) {
            atomicAdd(&st->n_acc, 1ull);
            const float u0 = o.u0, u2 = u0 * u0;
            atomicAdd(&st->hist[hist_bin(u0, __ldg(&P->hist_a), __ldg(&P->hist_b))], 1ull);
            atomicAdd(&st->exc[exc_bin(u0, __ldg(&P->exc_a))], 1ull);
            atomicAdd(&st->q[0], (unsigned long long)__float2ll_rn(u0 * kQ1));
            atomicAdd(&st->q[1], (unsigned long long)__float2ll_rn(u2 * kQ2));
            atomicAdd(&st->q[2], (unsigned long long)__float2ll_rn(u2 * u0 * kQ3));
            atomicAdd(&st->q[3], (unsigned long long)__float2ll_rn(u2 * u2 * kQ4));
            slot = atomicAdd(B.ring_count, 1ull);
            if (slot >= B.ring_cap) atomicAdd(&st->n_dropped, 1ull);
        }
        slot = __shfl_sync(0xffffffffu, slot, 0);
        unsigned char *rec = slot < B.ring_cap ? B.ring + slot * B.rec_bytes : nullptr;
        float *xh = rec ? reinterpret_cast<float *>(rec + 32) : nullptr;
        for (int m = lane; m < K; m += 32) {
            const double2 v = sx[m];
            const float xf = (float)(v.x * inv), yf = (float)(v.y * inv);
            atomicAdd(&st->spec[m], (unsigned long long)__float2ull_rn(fmaf(xf, xf, yf * yf) * kSpecScale));
            if (xh) {
                xh[m] = xf;
                xh[K + m] = yf;
            }
        }
        if (rec && lane == 0) {
            *reinterpret_cast<unsigned long long *>(rec) = it.idx;
            uint32_t *h = reinterpret_cast<uint32_t *>(rec + 8);
            h[0] = it.point;
            h[1] = 1u | (o.near ? 2u : 0u);
            float *f = reinterpret_cast<float *>(rec + 16);
            f[0] = o.H2;
            f[1] = o.H3;
            f[2] = o.u0;
            f[3] = (float)o.delta;
        }
    }
}

template <bool UNIF, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
    k_sample_warp(const __grid_constant__ DevBufs B, const __grid_constant__ RunArgs A, uint32_t k0, uint32_t k1) {
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) float2 s_slabs[];
    __shared__ WShared sh;
    __shared__ uint32_t s_hist[kHistBins];
    __shared__ uint32_t s_exc[kExcBins];
    __shared__ unsigned long long s_q[4];
    __shared__ unsigned long long s_spec[kWK];
    __shared__ uint32_t s_cnt[4];  // accepted, envelope violations, dropped, fallbacks
    __shared__ uint32_t s_maxd;
    __shared__ uint32_t s_chunk;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, ql = lane & 3;
    wshared_init(sh, s_slabs, NW, tid, NT);
    for (int e = tid; e < kHistBins; e += NT) s_hist[e] = 0;
    for (int e = tid; e < kWK; e += NT) s_spec[e] = 0ull;
    if (tid < kExcBins) s_exc[tid] = 0;
    if (tid < 4) {
        s_q[tid] = 0ull;
        s_cnt[tid] = 0;
    }
    if (tid == 0) s_maxd = 0;
    float2 *sv = s_slabs + warp * kWarpWords;
    const uint32_t total = A.chunk_prefix[A.n_points];
    const unsigned long long t0 = A.deadline_ns ? globaltimer_ns() : 0ull;

    for (;;) {
        if (tid == 0) {
            uint32_t c = atomicAdd(&B.counters[0], 1u);
            if (A.deadline_ns && c < total && globaltimer_ns() - t0 > A.deadline_ns) {
                atomicOr(B.status, kStatusDeadline);
                c = total;
            }
            s_chunk = c;
        }
        __syncthreads();
        const uint32_t c = s_chunk;
        if (c >= total) break;
        int p = 0;
        while (p + 1 < A.n_points && A.chunk_prefix[p + 1] <= c) ++p;
        const unsigned long long local = (unsigned long long)(c - A.chunk_prefix[p]) * A.chunk;
        const unsigned long long left = A.count[p] - local;
        const uint32_t n_here = left < A.chunk ? (uint32_t)left : A.chunk;
        const unsigned long long base = A.idx0[p] + local;
        const PointConst *P = B.pts + p;
        for (int e = tid; e < kWK; e += NT) {
            sh.sig[e] = __ldg(&P->sigma[e]);
            sh.act[e] = __ldg(&P->act[e]);
        }
        const Scal sc = load_scal(P);
        __syncthreads();

        float maxd = -INFINITY;
        WHeads heads;
        heads.make((uint32_t)(base >> 32), sc.pid, A.rk.k, lane);
        unsigned long long spec[kWK / 32] = {0ull, 0ull, 0ull, 0ull}, qsum[4] = {0ull, 0ull, 0ull, 0ull};
        for (uint32_t i0 = (uint32_t)warp * kWQ; i0 < n_here; i0 += (uint32_t)NW * kWQ) {
            const uint32_t left_here = n_here - i0, vmask = left_here < kWQ ? (1u << left_here) - 1u : (1u << kWQ) - 1u;
            const WEval ev = warp_batch<UNIF>(
                sv, sh.tw, sh.sig, sh.act, sc.K, [&](int q) { return base + i0 + (unsigned)q; }, vmask, heads, sc.pid,
                A.rk.k, lane);
            const unsigned long long idx = base + i0 + (unsigned)ql;
            const uint32_t lq = (uint32_t)idx, hq = (uint32_t)(idx >> 32);
            const uint32_t wa = PhiloxRow(lq, hq, sc.pid, A.rk.k).block((uint32_t)((sc.K + 1) / 2)).x;
            const Fast f = warp_eval<UNIF>(ev, sc, wa);
            const bool valid = lane < kWQ && ((vmask >> lane) & 1u);
            const bool tail = ev.tail || wa < kTailBucket;
            bool defer = valid && (fabsf(f.d) < f.guard || tail);
            if (valid && !tail) maxd = fmaxf(maxd, f.delta);

            const unsigned md = __ballot_sync(0xffffffffu, defer);
            if (md) {
                const int leader = __ffs(md) - 1;
                uint32_t slot0 = 0;
                if (lane == leader) slot0 = atomicAdd(&B.counters[1], (uint32_t)__popc(md));
                slot0 = __shfl_sync(0xffffffffu, slot0, leader);
                if (defer) {
                    const uint32_t slot = slot0 + __popc(md & ((1u << lane) - 1u));
                    if (slot < B.refine_cap) {
                        RefineItem it;
                        it.idx = ((unsigned long long)hq << 32) | lq;
                        it.point = (uint32_t)p;
                        it.pad = 0;
                        B.refine[slot] = it;
                    } else {  // queue full: decide in FP32 and flag the run
                        atomicOr(B.status, kStatusRefineOverflow);
                        atomicAdd(&s_cnt[3], 1u);
                        defer = false;
                    }
                }
            }
            const bool acc = valid && !defer && f.d < 0.f;
            if (valid && !defer && f.delta > 0.f) atomicAdd(&s_cnt[1], 1u);

            unsigned ma = __ballot_sync(0xffffffffu, acc);
            if (ma) {
                // one slot range for the batch; the lane of an accepted draw
                // tallies u(0) and writes the header, then the warp takes the
                // draws in turn, four modes per lane, the spectrum summed in
                // registers until the end of the chunk
                unsigned long long slot0 = 0;
                if (lane == 0) {
                    slot0 = atomicAdd(B.ring_count, (unsigned long long)__popc(ma));
                    atomicAdd(&s_cnt[0], (uint32_t)__popc(ma));
                }
                slot0 = __shfl_sync(0xffffffffu, slot0, 0);
                unsigned char *rec = nullptr;
                if (acc) {
                    const float u0 = sc.u0s * ev.u0raw * f.inv, u2 = u0 * u0;
                    atomicAdd(&s_hist[hist_bin(u0, sc.ha, sc.hb)], 1u);
                    atomicAdd(&s_exc[exc_bin(u0, sc.ea)], 1u);
                    qsum[0] += (unsigned long long)fixed_ll(u0 * kQ1);
                    qsum[1] += (unsigned long long)fixed_ll(u2 * kQ2);
                    qsum[2] += (unsigned long long)fixed_ll(u2 * u0 * kQ3);
                    qsum[3] += (unsigned long long)fixed_ll(u2 * u2 * kQ4);
                    const unsigned long long slot = slot0 + __popc(ma & ((1u << lane) - 1u));
                    if (slot < B.ring_cap) {
                        rec = B.ring + slot * B.rec_bytes;
                        write_header(rec, ((unsigned long long)hq << 32) | lq, (uint32_t)p, 0u, sc.E0 * f.S,
                                     sc.h3s * f.T, u0, f.delta);  // (H3 and log f/(Mg) again below)
                    } else {
                        atomicAdd(&s_cnt[2], 1u);
                    }
                }
                do {
                    const int q = __ffs(ma) - 1;
                    ma &= ma - 1;
                    const float inv = __shfl_sync(0xffffffffu, f.inv, q);
                    float *xh = reinterpret_cast<float *>(
                        __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(rec), q));
                    const float sc2 = (inv * inv) * kSpecScale;
                    if (xh) {  // the same in every lane
                        WEval out = ev;
                        out.T = fold_T(sv + q * kWS, sc.K, lane);
                        if (lane == q) {
                            const Fast g = warp_eval<UNIF>(out, sc, wa);
                            xh[5] = sc.h3s * g.T;
                            xh[7] = g.delta;
                        }
                    }
#pragma unroll
                    for (int cc = 0; cc < kWK / 32; ++cc) {
                        const int m = lane + 32 * cc;
                        if (m < sc.K) {
                            const float2 v = sv[q * kWS + m];
                            // (below 2^28: the 32-bit conversion; the 64-bit one runs on the FP64 pipe)
                            spec[cc] += __float2uint_rn(fmaf(v.x, v.x, v.y * v.y) * sc2);
                            if (xh) {
                                xh[8 + m] = v.x * inv;
                                xh[8 + sc.K + m] = v.y * inv;
                            }
                        }
                    }
                } while (ma);
            }
            __syncwarp();  // the next batch overwrites the slab
        }
        // chunk done: flush this CTA's partials into the point's StatBlock
#pragma unroll
        for (int cc = 0; cc < kWK / 32; ++cc)
            if (spec[cc]) atomicAdd(&s_spec[lane + 32 * cc], spec[cc]);
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (qsum[e]) atomicAdd(&s_q[e], qsum[e]);
        uint32_t key = fkey(maxd);
        key = __reduce_max_sync(0xffffffffu, key);
        if (lane == 0 && maxd > -INFINITY) atomicMax(&s_maxd, key);
        __syncthreads();
        StatBlock *st = B.stats + p;
        for (int e = tid; e < kHistBins; e += NT) {
            if (s_hist[e]) {
                atomicAdd(&st->hist[e], (unsigned long long)s_hist[e]);
                s_hist[e] = 0;
            }
        }
        if (tid < kExcBins && s_exc[tid]) {
            atomicAdd(&st->exc[tid], (unsigned long long)s_exc[tid]);
            s_exc[tid] = 0;
        }
        if (tid < 4 && s_q[tid]) {
            atomicAdd(&st->q[tid], s_q[tid]);
            s_q[tid] = 0ull;
        }
        for (int e = tid; e < kWK; e += NT) {
            if (s_spec[e]) {
                atomicAdd(&st->spec[e], s_spec[e]);
                s_spec[e] = 0ull;
            }
        }
        if (tid == 0) {
            atomicAdd(&st->n_prop, (unsigned long long)n_here);
            if (s_cnt[0]) atomicAdd(&st->n_acc, (unsigned long long)s_cnt[0]);
            if (s_cnt[1]) atomicAdd(&st->n_viol, (unsigned long long)s_cnt[1]);
            if (s_cnt[2]) atomicAdd(&st->n_dropped, (unsigned long long)s_cnt[2]);
            if (s_cnt[3]) atomicAdd(&st->n_fallback, (unsigned long long)s_cnt[3]);
            if (s_maxd) atomicMax(&st->maxd_key, (unsigned long long)s_maxd);
            s_cnt[0] = s_cnt[1] = s_cnt[2] = s_cnt[3] = 0;
            s_maxd = 0;
        }
        __syncthreads();
    }
}

// Replay: per-proposal outputs of listed indices, four per warp (the same
// batch code as the sampler).  out row: [delta, lnU, accept, flags, H2, H3,
// u0, S, xhat(2K)].
constexpr int kReplayWarps = 4;

template <bool UNIF>
__global__ void __launch_bounds__(32 * kReplayWarps) k_replay_warp(const PointConst *P, const unsigned long long *idx,
                                                                   unsigned long long n, uint32_t k0, uint32_t k1,
                                                                   double *out) {
    __shared__ WShared sh;
    __shared__ __align__(16) float2 s_slabs[kReplayWarps * kWarpWords];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, ql = lane & 3;
    wshared_init(sh, s_slabs, kReplayWarps, tid, 32 * kReplayWarps);
    for (int e = tid; e < kWK; e += 32 * kReplayWarps) {
        sh.sig[e] = P->sigma[e];
        sh.act[e] = P->act[e];
    }
    __syncthreads();
    const Scal sc = load_scal(P);
    const int K = sc.K;
    const unsigned long long b0 = ((unsigned long long)blockIdx.x * kReplayWarps + warp) * kWQ;
    if (b0 >= n) return;  // whole warps leave together
    float2 *sv = s_slabs + warp * kWarpWords;
    // the FP64 state of a proposal takes the place of the transform
    double2 *sx = reinterpret_cast<double2 *>(sv + kWQ * kWS);
    static_assert(sizeof(double2) * kWK <= sizeof(float2) * kWQ * kWB, "the FP64 state fits the transform's words");
    const uint32_t vmask = n - b0 < kWQ ? (1u << (n - b0)) - 1u : (1u << kWQ) - 1u;
    uint32_t rk[20];
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        rk[2 * r] = k0 + (uint32_t)r * 0x9E3779B9u;
        rk[2 * r + 1] = k1 + (uint32_t)r * 0xBB67AE85u;
    }
    WHeads heads;
    heads.make((uint32_t)(idx[b0] >> 32), sc.pid, rk, lane);
    const WEval ev = warp_batch<UNIF>(
        sv, sh.tw, sh.sig, sh.act, K, [&](int q) { return idx[b0 + q]; }, vmask, heads, sc.pid, rk, lane);
    const unsigned long long iq = idx[b0 + ql < n ? b0 + ql : n - 1];
    const uint32_t lq = (uint32_t)iq, hq = (uint32_t)(iq >> 32);
    const uint32_t wa = accept_word(lq, hq, sc.pid, K, k0, k1);
    const Fast f = warp_eval<UNIF>(ev, sc, wa);
    const bool valid = lane < kWQ && ((vmask >> lane) & 1u);
    const bool slow = fabsf(f.d) < f.guard || ev.tail || wa < kTailBucket;
    const size_t rowlen = 8 + 2 * (size_t)K;
    // the outputs of the proposals decided in FP32, T by the double sum
    const unsigned mf = __ballot_sync(0xffffffffu, valid && !slow);
    WEval eo = ev;
    for (int q = 0; q < kWQ; ++q) {
        if (!((mf >> q) & 1u)) continue;
        const float T = fold_T(sv + q * kWS, K, lane);
        if (lane == q) eo.T = T;
    }
    if (valid && !slow) {
        const Fast g = warp_eval<UNIF>(eo, sc, wa);
        double *row = out + (b0 + lane) * rowlen;
        {
            row[0] = g.delta;
            row[1] = f.lnU;
            row[2] = f.d < 0.f ? 1.0 : 0.0;
            row[3] = 0.0;
            row[4] = sc.E0 * f.S;
            row[5] = sc.h3s * g.T;
            row[6] = sc.u0s * ev.u0raw * f.inv;
            row[7] = f.S;
        }
    }
    // the proposals of the FP64 pass, one after the other on the whole warp
    unsigned ms = __ballot_sync(0xffffffffu, valid && slow);
    while (ms) {
        const int q = __ffs(ms) - 1;
        ms &= ms - 1;
        const unsigned long long id =
            ((unsigned long long)__shfl_sync(0xffffffffu, hq, q) << 32) | __shfl_sync(0xffffffffu, lq, q);
        Out64 o;
        double inv;
        eval64_warp<UNIF>(P, id, k0, k1, sx, lane, o, inv);
        double *row = out + (b0 + q) * rowlen;
        if (lane == 0) {
            row[0] = o.delta;
            row[1] = o.lnU;
            row[2] = o.accept;
            row[3] = 1.0 + (o.near ? 2.0 : 0.0);
            row[4] = o.H2;
            row[5] = o.H3;
            row[6] = o.u0;
            row[7] = o.S;
        }
        for (int m = lane; m < K; m += 32) {
            const double2 v = sx[m];
            row[8 + m] = (float)(v.x * inv);
            row[8 + K + m] = (float)(v.y * inv);
        }
    }
    // projected state of the proposals decided in FP32, written by the warp
    for (int q = 0; q < kWQ; ++q) {
        if (!((mf >> q) & 1u)) continue;
        const float inv = __shfl_sync(0xffffffffu, f.inv, q);
        double *row = out + (b0 + q) * rowlen;
        for (int m = lane; m < K; m += 32) {
            const float2 v = sv[q * kWS + m];
            row[8 + m] = v.x * inv;
            row[8 + K + m] = v.y * inv;
        }
    }
}

}  // namespace

void triad_kernels_k128(TriadKernels *t) {
    t->main[0][0] = (const void *)k_sample_warp<false, 128, 1>;
    t->main[0][1] = (const void *)k_sample_warp<false, 256, 1>;
    t->main[0][2] = (const void *)k_sample_warp<false, 256, 2>;
    t->main[1][0] = (const void *)k_sample_warp<true, 128, 1>;
    t->main[1][1] = (const void *)k_sample_warp<true, 256, 1>;
    t->main[1][2] = (const void *)k_sample_warp<true, 256, 2>;
    t->sir[0] = t->sir[1] = nullptr;  // SIR runs use the one-thread form (K <= 64)
    t->refine[0] = (const void *)k_refine_warp<false>;
    t->refine[1] = (const void *)k_refine_warp<true>;
    t->refine_smem = 0;
    t->refine_threads = 128;
    t->refine_ctas = 4;
    t->replay[0] = (const void *)k_replay_warp<false>;
    t->replay[1] = (const void *)k_replay_warp<true>;
    t->replay_per_block = 32 * kReplayWarps / 32 * kWQ;
    t->xfer_bytes_per_thread = kWarpWords * (int)sizeof(float2) / 32;  // the warps' slabs
    t->n_variants = 3;
}

}  // namespace tkdv
