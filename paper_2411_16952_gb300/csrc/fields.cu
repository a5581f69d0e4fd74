// Largest surface displacement of accepted fields on the 2K-point grid of
// Sec. V.D (the "1-in-m event" of Figs. 8-11 is the field with the largest
// such maximum among m accepted fields).  An opt-in pass over the kept
// records: one warp per record, each lane a few grid points.
#include <cuda_runtime.h>

#include <algorithm>

#include "tkdv_internal.h"

namespace tkdv {

// u(xi_j) = u0s sum_k (xh_k cos k xi_j + xh_{K+k} sin k xi_j) (Eq. 8 with
// Eq. 16), xi_j = -pi + pi j / K, so cos k xi_j = (-1)^k cos(pi k j / K) and
// sin k xi_j = (-1)^k sin(pi k j / K); the phases come from a table of
// cos, sin (pi m / K), m = 0..2K-1, and index k j mod 2K.
__global__ void __launch_bounds__(128) k_field_max(const unsigned char *__restrict__ ring, unsigned long long rec_bytes,
                                                   unsigned long long n, int K,
                                                   const PointConst *__restrict__ pts,
                                                   const unsigned long long *__restrict__ list,
                                                   const unsigned long long *__restrict__ n_list, float *umax, int *jmax,
                                                   unsigned long long *idx) {
    // list: the records to take (n of them at most, *n_list listed), else the first n
    if (list) n = *n_list < n ? *n_list : n;
    __shared__ float s_c[2 * kKMax], s_s[2 * kKMax];
    const int G = 2 * K;
    for (int m = threadIdx.x; m < G; m += blockDim.x) {
        float sn, cs;
        sincospif((float)m / (float)K, &sn, &cs);
        s_c[m] = cs;
        s_s[m] = sn;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const unsigned long long warps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    for (unsigned long long r = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < n;
         r += warps) {
        const unsigned char *rec = ring + (list ? list[r] : r) * rec_bytes;
        const uint32_t point = *reinterpret_cast<const uint32_t *>(rec + 8);
        const float *xh = reinterpret_cast<const float *>(rec + 32);
        float best = -INFINITY;
        int bj = 0;
        for (int j = lane; j < G; j += 32) {
            float acc = 0.f;
            int id = 0;
            for (int k = 1; k <= K; ++k) {
                id += j;
                if (id >= G) id -= G;
                const float t = fmaf(__ldg(&xh[k - 1]), s_c[id], __ldg(&xh[K + k - 1]) * s_s[id]);
                acc = (k & 1) ? acc - t : acc + t;
            }
            if (acc > best) {
                best = acc;
                bj = j;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
            if (ob > best || (ob == best && oj < bj)) {
                best = ob;
                bj = oj;
            }
        }
        if (lane == 0) {
            umax[r] = __ldg(&pts[point].u0s) * best;
            jmax[r] = bj;
            if (idx) idx[r] = *reinterpret_cast<const unsigned long long *>(rec);
        }
    }
}

cudaError_t launch_field_max(const unsigned char *ring, unsigned long long rec_bytes, unsigned long long n, int K,
                             const PointConst *pts, float *umax, int *jmax, cudaStream_t st) {
    if (!n) return cudaSuccess;
    const unsigned long long blocks = std::min<unsigned long long>((n + 3) / 4, 65535ull * 16);
    return launch_kernel(k_field_max, (unsigned)blocks, 128, 0, st, ring, rec_bytes, n, K, pts, nullptr, nullptr, umax, jmax,
                         nullptr);
}

// ---- the 1-in-m event ----------------------------------------------------------
// The extreme field of an ensemble is the one with the largest maximum among
// the first m accepted fields of a point by proposal index (ties of the index,
// from runs with several seeds, by ring position; ties of the maximum, the
// first).  The ring is unordered, so the m smallest (index, position) pairs
// are found by a radix selection on the device, the maxima are taken of those
// m fields only, and one record goes to the host.
//
// What bounds it: launches, a dozen in a row without a host wait (about 60 us);
// each pass reads 8 bytes a record (2.4 MB at 300,000 records).  Decoding all
// records on the host instead took 45 ms at 300,000 records of 32 modes, one
// copy of 86 MB and four of its columns.
namespace {

constexpr int kDigit = 11, kBins = 1 << kDigit;

struct SelState {
    unsigned long long n_match;  // records of the point
    unsigned long long want;     // still to take within the current prefix
    unsigned long long prefix;   // digits fixed so far
    unsigned long long thr;      // the largest index taken
    uint32_t done;               // blocks of the current pass that have finished
    unsigned long long n_list;   // fields listed
    uint32_t hist[kBins];
};

__global__ void k_sel_init(SelState *s, unsigned long long m) {
    for (int b = threadIdx.x; b < kBins; b += blockDim.x) s->hist[b] = 0;
    if (threadIdx.x == 0) {
        s->n_match = 0;
        s->want = m;
        s->prefix = 0;
        s->thr = 0;
        s->done = 0;
        s->n_list = 0;
    }
}

// (index, ring position) of the point's records, in any order.
__global__ void __launch_bounds__(256) k_sel_gather(const unsigned char *__restrict__ ring, unsigned long long rec_bytes,
                                                    unsigned long long n, uint32_t point, SelState *s,
                                                    unsigned long long *key, unsigned long long *pos) {
    const int lane = threadIdx.x & 31;
    const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long r0 = (unsigned long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); r0 < n; r0 += step) {
        const unsigned long long r = r0 + (unsigned)lane;
        bool in = false;
        unsigned long long idx = 0;
        if (r < n) {
            const uint4 h = __ldg(reinterpret_cast<const uint4 *>(ring + r * rec_bytes));  // idx, point, flags
            idx = ((unsigned long long)h.y << 32) | h.x;
            in = h.z == point;
        }
        const unsigned mk = __ballot_sync(0xffffffffu, in);
        if (!mk) continue;
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(&s->n_match, (unsigned long long)__popc(mk));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(mk & ((1u << lane) - 1u));
        if (in) {
            key[at] = idx;
            pos[at] = r;
        }
    }
}

// One digit of the selection: the values (the keys, or with POS the positions
// of the keys equal to thr) that share the prefix are counted by their digit;
// the last block to finish fixes the digit that holds the want-th value.
template <bool POS>
__global__ void __launch_bounds__(256) k_sel_pass(SelState *s, const unsigned long long *__restrict__ key,
                                                  const unsigned long long *__restrict__ pos, int shift, int first, int last) {
    __shared__ uint32_t sh[kBins];
    __shared__ bool s_last;
    for (int b = threadIdx.x; b < kBins; b += blockDim.x) sh[b] = 0;
    __syncthreads();
    const unsigned long long n = s->n_match, prefix = s->prefix, thr = s->thr;
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long k = key[i];
        if (POS && k != thr) continue;
        const unsigned long long v = POS ? pos[i] : k;
        if (first || (v >> (shift + kDigit)) == prefix) atomicAdd(&sh[(v >> shift) & (kBins - 1)], 1u);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kBins; b += blockDim.x)
        if (sh[b]) atomicAdd(&s->hist[b], sh[b]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&s->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    // sums of 8 bins per thread, then one thread walks the 256 sums and 8 bins
    __threadfence();
    uint32_t sum = 0;
    for (int e = 0; e < kBins / 256; ++e) sum += *(volatile uint32_t *)&s->hist[threadIdx.x * (kBins / 256) + e];
    sh[threadIdx.x] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long want = s->want;
        int g = 0;
        while (g < 255 && want > sh[g]) want -= sh[g++];
        int b = g * (kBins / 256);
        const int end = b + kBins / 256 - 1;
        while (b < end && want > *(volatile uint32_t *)&s->hist[b]) want -= *(volatile uint32_t *)&s->hist[b++];
        s->want = want;
        s->prefix = (first ? 0ull : prefix << kDigit) | (unsigned long long)b;
        s->done = 0;
        if (!POS && last) {
            s->thr = s->prefix;
            s->prefix = 0;
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kBins; e += blockDim.x) s->hist[e] = 0;
}

// The ring positions of the selected fields.
__global__ void __launch_bounds__(256) k_sel_list(SelState *s, const unsigned long long *__restrict__ key,
                                                  const unsigned long long *__restrict__ pos,
                                                  unsigned long long *list, unsigned long long cap) {
    const unsigned long long n = s->n_match, thr = s->thr, pthr = s->prefix;
    for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long k = key[i];
        if (k < thr || (k == thr && pos[i] <= pthr)) {
            const unsigned long long at = atomicAdd(&s->n_list, 1ull);
            if (at < cap) list[at] = pos[i];
        }
    }
}

}  // namespace

size_t extreme_scratch_bytes(unsigned long long n, unsigned long long m) {
    return sizeof(SelState) + 16 * n + 24 * m + 256;
}

cudaError_t launch_extreme(const unsigned char *ring, unsigned long long rec_bytes, unsigned long long n, int K,
                           const PointConst *pts, uint32_t point, unsigned long long m, void *scratch,
                           ExtremeBufs *out, cudaStream_t st) {
    static_assert(sizeof(SelState) % 16 == 0, "the arrays after the state are aligned");
    SelState *s = (SelState *)scratch;
    unsigned long long *key = (unsigned long long *)(s + 1), *pos = key + n, *list = pos + n, *idx = list + m;
    float *umax = (float *)(idx + m);
    int *jmax = (int *)(umax + m);
    *out = ExtremeBufs{&s->n_match, list, idx, umax, jmax};
    const unsigned blocks = (unsigned)std::min<unsigned long long>((n + 1023) / 1024, 608);
    cudaError_t e = launch_kernel(k_sel_init, 1, 256, 0, st, s, m);
    if (e == cudaSuccess) e = launch_kernel(k_sel_gather, blocks, 256, 0, st, ring, rec_bytes, n, point, s, key, pos);
    for (int d = 5; d >= 0 && e == cudaSuccess; --d)
        e = launch_kernel(k_sel_pass<false>, blocks, 256, 0, st, s, key, pos, d * kDigit, d == 5, d == 0);
    int digits = 1;
    while ((n - 1) >> (digits * kDigit)) ++digits;
    for (int d = digits - 1; d >= 0 && e == cudaSuccess; --d)
        e = launch_kernel(k_sel_pass<true>, blocks, 256, 0, st, s, key, pos, d * kDigit, d == digits - 1, d == 0);
    if (e == cudaSuccess) e = launch_kernel(k_sel_list, blocks, 256, 0, st, s, key, pos, list, m);
    const unsigned fb = (unsigned)std::min<unsigned long long>((m + 3) / 4, 65535ull * 16);
    if (e == cudaSuccess)
        e = launch_kernel(k_field_max, fb, 128, 0, st, ring, rec_bytes, m, K, pts, list, &s->n_list, umax, jmax, idx);
    return e;
}

}  // namespace tkdv
