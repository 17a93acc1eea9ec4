// Volume -> Gaussians (Sec. 4.1-4.3): transfer function and periodised 3D DWT
// (dwt.cu), adaptive coefficient filtering (Supp. Sec. 1) and the
// per-coefficient map (Eq. 22-24).  A setup step, run once per volume and TF.
//
// Selection, all on the device and over every subband in the same launches:
//   v = sqrt(((a0 a0 + a1 a1) + a2 a2) + a3 a3) in IEEE float32, rounded op by
//   op (explicit __fmul_rn/__fadd_rn/__fsqrt_rn, so the order is fixed);
//   the medians and the K-th largest value by radix select on the float bits (v >= 0
//   so the bits order like the values): three passes of 10 or 11 bits, no sort;
//   sigma = MAD / 0.6745 and T = lambda sigma in float32;
//   keep = v >= max(T, v_(K')) and v > 0.
// Kept coefficients are marked in a bit mask (raster order of each subband),
// whose counts are scanned, and mapped chunk by chunk to the P[14][capacity]
// layout.  The host waits for the number kept and for the end.  One launch a
// pass over all bands (one where every band is small, else six, and two for the
// marking and the map) instead of about 50 a band, and a map over the whole chip
// instead of one block a band (which took 350 ms on a 512^3 volume): with the
// DWT's kernels, vbm_build of 32^3 / 224 x 160 x 96 / 512^3 volumes 5.5 -> 0.13,
// 18.9 -> 0.34, 390 -> 3.9 ms (selection passes 0.09 of the second, 0.63 of the
// third).
#include <cmath>
#include <vector>

#include "vbm_internal.h"

namespace vbm {

namespace {

// ----------------------------------------------------------------- select

constexpr int kMaxBands = 64;            // 7 J + 1 with J <= 9
constexpr int kSelThreads = 1024;
constexpr int kTargets = 3;              // lower median rank, upper median rank, K-th largest
constexpr int kBins = 2048;              // bins of the widest digit
constexpr int kChunk = 8192;             // elements of one marking / mapping block
constexpr int kMarkThreads = 256;

struct Band {
    int j, o[3], ox, oy, oz, mx, my, mz;
    int64_t n;
};

// Where the subbands lie: element i (raster order) of band b is word voff[b] +
// i of the magnitude array (each band padded to whole 32-bit mask words), and
// pyramid element (oz + z, oy + y, ox + x).  chunk0 and blk0 are the first
// marking chunk and the first selection block of a band ([nb]: the totals).
struct BandTab {
    int nb;
    int ox[kMaxBands], oy[kMaxBands], oz[kMaxBands], mx[kMaxBands], my[kMaxBands];
    int64_t n[kMaxBands], voff[kMaxBands];
    double n_beta[kMaxBands];            // N^beta of the budget
    int chunk0[kMaxBands + 1], blk0[kMaxBands + 1];
};

// Budget of Supp. Sec. 1.1, evaluated on the device from the band energies.
struct Budget {
    double alpha_E, K_tot;
    int64_t min_per_band;
    float lambda;
};

// Running selections of one band.  rank: what is left of each target's rank
// inside its prefix; prefix: the digits found so far.
struct SubState {
    unsigned long long zeros[2];         // exact zeros among the magnitudes / the deviations
    long long rank[kTargets];
    uint32_t prefix[kTargets];
    uint32_t ticket;                     // blocks of the running pass that are done (wraps to 0)
    int none;                            // the budget is 0: nothing is kept
    float med, vk, thr;
};

__device__ __forceinline__ int band_of(const int *first, int nb, int blk)
{
    int b = 0;
    while (b < nb - 1 && blk >= first[b + 1]) b++;
    return b;
}

// Pyramid element of band element i.
__device__ __forceinline__ int64_t pyramid_index(const BandTab &t, int b, int64_t i, int nx, int ny, int &x, int &y,
                                                 int &z)
{
    const int64_t row = t.n[b] <= INT_MAX ? (int64_t)((uint32_t)i / (uint32_t)t.mx[b]) : i / t.mx[b];
    x = (int)(i - row * t.mx[b]);
    z = t.n[b] <= INT_MAX ? (int)((uint32_t)row / (uint32_t)t.my[b]) : (int)(row / t.my[b]);
    y = (int)(row - (int64_t)z * t.my[b]);
    return ((int64_t)(t.oz[b] + z) * ny + (t.oy[b] + y)) * nx + (t.ox[b] + x);
}

// Exclusive block scan of one count per thread; `total` is the block's sum.
template <int THREADS>
__device__ __forceinline__ uint32_t block_scan(uint32_t c, uint32_t *warp_sum, uint32_t &total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t incl = c;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    __syncthreads();                     // the last user of warp_sum is done
    if (lane == 31) warp_sum[w] = incl;
    __syncthreads();
    uint32_t base = 0;
    total = 0;
#pragma unroll
    for (int k = 0; k < THREADS / 32; k++) {
        const uint32_t ws = warp_sum[k];
        base += k < w ? ws : 0u;
        total += ws;
    }
    return base + incl - c;
}

// The three digits of a selection on the float bits (v >= 0, so the sign bit
// is 0 and the bits order like the values): bits 30-21, 20-10 and 9-0.
template <int DIGIT>
struct Digit {
    static constexpr int shift = DIGIT == 0 ? 21 : DIGIT == 1 ? 10 : 0;
    static constexpr int bits = DIGIT == 1 ? 11 : 10;
};

// Shared memory of a block that picks digits.
struct Pick {
    uint32_t sums[kTargets][32];
    uint32_t digit[kTargets], rest[kTargets], prefix[kTargets];
    long long rank[kTargets];
};

// The digit of each of N targets: the bin of its histogram (count(k, bin)) in
// which its rank falls; the rank becomes the rest inside that bin and the digit
// joins the prefix.  All kSelThreads threads; the targets share the barriers.
template <int BITS, int N, typename F>
__device__ __forceinline__ void pick_digits(Pick &s, F count)
{
    constexpr int PER = (1 << BITS) / kSelThreads;
    static_assert(PER >= 1 && kSelThreads == 1024, "whole bins a thread, one warp sum a lane");
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t c[N][PER], mine[N], incl[N];
#pragma unroll
    for (int k = 0; k < N; k++) {
        mine[k] = 0;
#pragma unroll
        for (int i = 0; i < PER; i++) mine[k] += c[k][i] = count(k, threadIdx.x * PER + i);
        incl[k] = mine[k];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl[k], off);
            if (lane >= off) incl[k] += y;
        }
        if (lane == 31) s.sums[k][w] = incl[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < N; k++) {
        const uint32_t before = __reduce_add_sync(0xffffffffu, lane < w ? s.sums[k][lane] : 0u);
        long long at = s.rank[k] - (long long)(before + incl[k] - mine[k]);
        if (at >= 0 && at < (long long)mine[k]) {
            int i = 0;
            while (i < PER - 1 && at >= (long long)c[k][i]) at -= c[k][i++];
            s.digit[k] = (uint32_t)(threadIdx.x * PER + i);
            s.rest[k] = (uint32_t)at;
        }
    }
    __syncthreads();
    if (threadIdx.x < N) {
        const int k = threadIdx.x;
        s.rank[k] = s.rest[k];
        s.prefix[k] = (s.prefix[k] << BITS) | s.digit[k];
    }
    __syncthreads();
}

// The budget of band b (Supp. Sec. 1.1): K = max(min_per_band, floor(K_tot S /
// sum S)), S = E^alpha N^beta, in thread 0's result.  All threads call it;
// share: kMaxBands doubles.  Double precision is slow here, so only the
// powers' threads and one adder use it.
__device__ __forceinline__ int64_t band_budget(const BandTab &t, const Budget &bud, const double *E, int b,
                                               double *share)
{
    if (threadIdx.x < (unsigned)t.nb) share[threadIdx.x] = pow(__ldcg(E + threadIdx.x), bud.alpha_E) * t.n_beta[threadIdx.x];
    __syncthreads();
    if (threadIdx.x != 0) return 0;
    double sum = 0.0;
    for (int k = 0; k < t.nb; k++) sum += share[k];
    const double mine = sum > 0 ? bud.K_tot * share[b] / sum : 0.0;
    return max(bud.min_per_band, (int64_t)floor(mine));
}

// The median of n values from its lower and upper middle value.
__device__ __forceinline__ float median_of(int64_t n, uint32_t lower, uint32_t upper)
{
    const float a = __uint_as_float(lower), c = __uint_as_float(upper);
    return (n & 1) ? c : __fmul_rn(__fadd_rn(a, c), 0.5f);
}

// Keep v >= max(T, v_(K')), K' = min(K, #{v >= T}): where fewer than K values
// reach T, v_(K) < T and the maximum is T itself, the same set.
__device__ __forceinline__ float threshold(float mad, float lambda, bool none, float vk)
{
    const float T = __fmul_rn(lambda, __fdiv_rn(mad, 0.6745f));
    return none || T != T ? __int_as_float(0x7f800000) : fmaxf(T, vk);
}

// Bands of at most kSmallBand elements: one block holds the band in registers
// and runs all six digit passes beside the larger bands' first one (a pass over
// 15 such bands cost 10 us as a launch of its own, nearly all of it latency).
constexpr int kSmallPer = 8;
constexpr int kSmallBand = kSmallPer * kSelThreads;

template <int DIGIT, int N>
__device__ __forceinline__ void small_digit(Pick &s, uint32_t (&h)[kTargets][kBins], uint32_t *zeros,
                                            const float (&x)[kSmallPer], int n)
{
    using D = Digit<DIGIT>;
    constexpr int NB = 1 << D::bits, NT = DIGIT == 0 ? 1 : N;
    const int tid = threadIdx.x;
#pragma unroll
    for (int k = 0; k < NT; k++)
        for (int i = tid; i < NB; i += kSelThreads) h[k][i] = 0;
    if (DIGIT == 0 && tid == 0) *zeros = 0;
    uint32_t p[N];
#pragma unroll
    for (int k = 0; k < N; k++) p[k] = s.prefix[k];
    __syncthreads();
    uint32_t zero = 0;
#pragma unroll
    for (int e = 0; e < kSmallPer; e++) {
        if (tid + e * kSelThreads >= n) continue;
        const uint32_t bits = __float_as_uint(x[e]);
        if (bits == 0) {
            zero++;
            continue;
        }
        const uint32_t d = (bits >> D::shift) & (NB - 1), pre = bits >> (D::shift + D::bits);
        if (DIGIT == 0) {
            atomicAdd(&h[0][d], 1u);
        } else {
#pragma unroll
            for (int k = 0; k < N; k++) {            // into the first target of its prefix
                if (pre != p[k]) continue;
                atomicAdd(&h[k][d], 1u);
                break;
            }
        }
    }
    if (DIGIT == 0) {
        zero = __reduce_add_sync(0xffffffffu, zero);
        if ((tid & 31) == 0 && zero) atomicAdd(zeros, zero);
    }
    __syncthreads();
    const uint32_t z = *zeros;
    pick_digits<D::bits, N>(s, [&](int k, int bin) {
        int src = 0;
        if (DIGIT > 0)
            while (p[src] != p[k]) src++;
        return h[src][bin] + (bin == 0 && p[k] == 0 ? z : 0u);
    });
}

__device__ void select_small(const float *__restrict__ v, const BandTab &t, const Budget &bud,
                             const double *__restrict__ E, SubState *__restrict__ st, int b,
                             uint32_t (&h)[kTargets][kBins], double *share, Pick &s, uint32_t *zeros)
{
    const int tid = threadIdx.x;
    const int n = (int)t.n[b];
    float x[kSmallPer];
#pragma unroll
    for (int e = 0; e < kSmallPer; e++)
        x[e] = tid + e * kSelThreads < n ? v[t.voff[b] + tid + e * kSelThreads] : 0.f;
    const int64_t K = band_budget(t, bud, E, b, share);
    if (tid == 0) {
        s.rank[0] = (n - 1) / 2;                     // the middle value, or the lower one of an even count
        s.rank[1] = n / 2;
        s.rank[2] = n - min(max(K, (int64_t)1), (int64_t)n);
        s.prefix[0] = s.prefix[1] = s.prefix[2] = 0;
    }
    __syncthreads();
    small_digit<0, 3>(s, h, zeros, x, n);
    small_digit<1, 3>(s, h, zeros, x, n);
    small_digit<2, 3>(s, h, zeros, x, n);
    const float med = median_of(n, s.prefix[0], s.prefix[1]), vk = __uint_as_float(s.prefix[2]);
    __syncthreads();
    if (tid == 0) {
        s.rank[0] = (n - 1) / 2;
        s.rank[1] = n / 2;
        s.prefix[0] = s.prefix[1] = 0;
    }
#pragma unroll
    for (int e = 0; e < kSmallPer; e++) x[e] = fabsf(__fsub_rn(x[e], med));
    __syncthreads();
    small_digit<0, 2>(s, h, zeros, x, n);
    small_digit<1, 2>(s, h, zeros, x, n);
    small_digit<2, 2>(s, h, zeros, x, n);
    if (tid == 0) st[b].thr = threshold(median_of(n, s.prefix[0], s.prefix[1]), bud.lambda, K <= 0, vk);
}

// One radix-select pass over every larger band at once: digit DIGIT of the magnitudes
// (DEV = false: both median ranks and the K-th largest in the same pass) or of
// their absolute deviations from the median (DEV = true: both median ranks),
// which are formed on the fly.  A block counts one band's digits in shared
// memory and adds them to the band's histogram; the band's last block picks
// the digits, clears the histogram for the next pass and, after the third
// digit, forms the median (the mean of the two middle values of an even
// count) or the threshold.
//
// Bound by reading the magnitudes (4 bytes an element a pass).  Wide digits
// keep the passes at three a selection; the first digit (sign-free exponent
// and two mantissa bits) falls into few bins, so its counts are kept in eight
// copies, one per lane mod 8, and exact zeros (empty space: often most of a
// volume) are counted in registers and left out of every histogram.
template <int DIGIT, bool DEV>
__global__ void __launch_bounds__(kSelThreads) k_select_pass(const float *__restrict__ v,
                                                             const __grid_constant__ BandTab t,
                                                             const __grid_constant__ Budget bud,
                                                             const double *__restrict__ E, SubState *__restrict__ st,
                                                             uint32_t *__restrict__ hist)
{
    using D = Digit<DIGIT>;
    constexpr int NB = 1 << D::bits;
    constexpr int NT = DIGIT == 0 ? 1 : DEV ? 2 : 3;             // histograms
    constexpr int COPIES = DIGIT == 0 ? 8 : 1;
    constexpr int WORDS = NT * NB * COPIES;
    __shared__ uint32_t h[WORDS];
    __shared__ Pick pick;
    __shared__ double share[kMaxBands];
    __shared__ uint32_t s_last;
    const int tid = threadIdx.x;
    if constexpr (DIGIT == 0 && !DEV) {
        static_assert(WORDS >= kTargets * kBins, "a small band's histograms fit");
        const int small = (int)blockIdx.x - t.blk0[t.nb];        // the blocks beyond the passes': one a band
        if (small >= 0) {
            if (t.n[small] <= kSmallBand)
                select_small(v, t, bud, E, st, small, reinterpret_cast<uint32_t(&)[kTargets][kBins]>(h), share, pick,
                             &s_last);
            return;
        }
    }
    const int b = band_of(t.blk0, t.nb, blockIdx.x);
    SubState *sb = st + b;
    uint32_t *gh = hist + (int64_t)b * kTargets * kBins;
    for (int i = tid; i < WORDS; i += kSelThreads) h[i] = 0;
    __syncthreads();
    const uint32_t p0 = sb->prefix[0], p1 = sb->prefix[1], p2 = sb->prefix[2];
    const float med = DEV ? sb->med : 0.f;
    uint32_t zeros = 0;
    auto count = [&](float val) {
        const float x = DEV ? fabsf(__fsub_rn(val, med)) : val;
        const uint32_t bits = __float_as_uint(x);
        if (bits == 0) {
            zeros++;
            return;
        }
        const uint32_t d = (bits >> D::shift) & (NB - 1);
        if constexpr (DIGIT == 0) {
            atomicAdd(&h[d * COPIES + (tid & (COPIES - 1))], 1u);
        } else {
            const uint32_t p = bits >> (D::shift + D::bits);
            if (p == p0) atomicAdd(&h[d], 1u);
            else if (p == p1) atomicAdd(&h[NB + d], 1u);         // where it left the lower rank's prefix
            if (NT == 3 && p == p2 && p2 != p0 && p2 != p1) atomicAdd(&h[(NT - 1) * NB + d], 1u);
        }
    };
    // this block's share of the band, in whole float4 (bands start on 128-byte boundaries)
    const int64_t quads = t.n[b] >> 2;
    const int nblk = t.blk0[b + 1] - t.blk0[b], blk = blockIdx.x - t.blk0[b];
    const int64_t q0 = quads * blk / nblk, q1 = quads * (blk + 1) / nblk;
    const float4 *v4 = reinterpret_cast<const float4 *>(v + t.voff[b]);
    int64_t q = q0 + tid;
    for (; q + 3 * kSelThreads < q1; q += 4 * kSelThreads) {
        float4 a[4];
#pragma unroll
        for (int u = 0; u < 4; u++) a[u] = v4[q + u * kSelThreads];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            count(a[u].x);
            count(a[u].y);
            count(a[u].z);
            count(a[u].w);
        }
    }
    for (; q < q1; q += kSelThreads) {
        const float4 a = v4[q];
        count(a.x);
        count(a.y);
        count(a.z);
        count(a.w);
    }
    if (blk == nblk - 1 && 4 * quads + tid < t.n[b]) count(v[t.voff[b] + 4 * quads + tid]);
    if constexpr (DIGIT == 0) {
        zeros = __reduce_add_sync(0xffffffffu, zeros);
        if ((tid & 31) == 0 && zeros) atomicAdd(&sb->zeros[DEV], (unsigned long long)zeros);
    }
    __syncthreads();
    for (int i = tid; i < NT * NB; i += kSelThreads) {
        uint32_t c = 0;
#pragma unroll
        for (int k = 0; k < COPIES; k++) c += h[i * COPIES + k];
        if (c) atomicAdd(&gh[(i / NB) * kBins + (i & (NB - 1))], c);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicInc(&sb->ticket, (uint32_t)nblk - 1) == (uint32_t)nblk - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // ---- the band's last block: pick the digits
    const int64_t n = t.n[b];
    const uint32_t n_zero = (uint32_t)__ldcg(&sb->zeros[DEV]);
    constexpr int N = DEV ? 2 : kTargets;
    int64_t K = 0;
    if (DIGIT == 0 && !DEV) K = band_budget(t, bud, E, b, share);
    if (tid == 0) {
        if (DIGIT == 0) {
            pick.rank[0] = (n - 1) / 2;      // the middle value, or the lower one of an even count
            pick.rank[1] = n / 2;
            pick.rank[2] = n - min(max(K, (int64_t)1), n);
            if (!DEV) sb->none = K <= 0;
        }
        for (int k = 0; k < N; k++) {
            if (DIGIT > 0) pick.rank[k] = sb->rank[k];
            pick.prefix[k] = DIGIT > 0 ? sb->prefix[k] : 0u;
        }
    }
    __syncthreads();
    uint32_t old[N];
#pragma unroll
    for (int k = 0; k < N; k++) old[k] = pick.prefix[k];
    pick_digits<D::bits, N>(pick, [&](int k, int bin) {
        // the histogram that counted this target's prefix
        const int src = DIGIT == 0 || old[k] == old[0] ? 0 : old[k] == old[1] ? 1 : 2;
        return __ldcg(&gh[src * kBins + bin]) + (bin == 0 && old[k] == 0 ? n_zero : 0u);
    });
    for (int i = tid; i < kTargets * kBins; i += kSelThreads) gh[i] = 0;
    if (tid >= N) return;
    sb->rank[tid] = pick.rank[tid];
    sb->prefix[tid] = pick.prefix[tid];
    if (DIGIT == 2 && tid == 0) {
        const float m = median_of(n, pick.prefix[0], pick.prefix[1]);
        if (!DEV) {
            sb->med = m;
            sb->vk = __uint_as_float(pick.prefix[2]);
        } else {
            sb->thr = threshold(m, bud.lambda, sb->none, sb->vk);
        }
    }
}

// ------------------------------------------------------- marking and map

// One bit per band element, set where the coefficient is kept (v >= threshold
// and v > 0), and each chunk's count; the grid's last block turns the counts
// into the chunks' first output columns and the total.  keep, if given,
// receives one byte per pyramid element.
__global__ void __launch_bounds__(kMarkThreads) k_mark(const float *__restrict__ v, const __grid_constant__ BandTab t,
                                                       int nx, int ny, const SubState *__restrict__ st,
                                                       uint32_t *__restrict__ mask, uint32_t *__restrict__ count,
                                                       int64_t *__restrict__ first, int64_t *__restrict__ total,
                                                       uint32_t *__restrict__ ticket, uint8_t *__restrict__ keep)
{
    constexpr int U = 8;                                  // words of a warp, loaded together
    __shared__ uint32_t s_count, s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_count = 0;
    __syncthreads();
    const int b = band_of(t.chunk0, t.nb, blockIdx.x);
    const int64_t i0 = (int64_t)(blockIdx.x - t.chunk0[b]) * kChunk, n = t.n[b];
    const float thr = st[b].thr;
    const float *vb = v + t.voff[b];
    uint32_t mine = 0;
    for (int w0 = warp * U; w0 < kChunk / 32; w0 += kMarkThreads / 32 * U) {
        float x[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t i = i0 + (w0 + u) * 32 + lane;
            x[u] = i < n ? vb[i] : 0.f;
        }
        uint32_t word = 0;
#pragma unroll
        for (int u = 0; u < U; u++) {
            const uint32_t bal = __ballot_sync(0xffffffffu, x[u] >= thr && x[u] > 0.f);
            word = lane == u ? bal : word;
        }
        if (lane < U && i0 + (w0 + lane) * 32 < n) {
            mask[(t.voff[b] + i0) / 32 + w0 + lane] = word;
            mine += __popc(word);
        }
        if (keep) {
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int64_t i = i0 + (w0 + u) * 32 + lane;
                int cx, cy, cz;
                if (i < n) keep[pyramid_index(t, b, i, nx, ny, cx, cy, cz)] = x[u] >= thr && x[u] > 0.f;
            }
        }
    }
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0) atomicAdd(&s_count, mine);
    __syncthreads();
    if (tid == 0) {
        count[blockIdx.x] = s_count;
        __threadfence();
        s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    __shared__ uint32_t warp_sum[kMarkThreads / 32];
    constexpr int PER = 16;
    int64_t run = 0;
    for (int c0 = 0; c0 < (int)gridDim.x; c0 += kMarkThreads * PER) {
        uint32_t c[PER], sum = 0, all;
#pragma unroll
        for (int k = 0; k < PER; k++) {
            const int i = c0 + tid * PER + k;
            c[k] = i < (int)gridDim.x ? __ldcg(count + i) : 0u;
            sum += c[k];
        }
        int64_t at = run + block_scan<kMarkThreads>(sum, warp_sum, all);
#pragma unroll
        for (int k = 0; k < PER; k++) {
            const int i = c0 + tid * PER + k;
            if (i < (int)gridDim.x) first[i] = at;
            at += c[k];
        }
        run += all;
    }
    if (tid == 0) *total = run;
}

struct MapEntry {
    float u[3];
    float w;
    float log_scale[3];
    float quat[4];
    float s;        // 2^{-3j/2} or 1
    int j;
};

struct MapTab {
    MapEntry e[kMaxBands];
};

// The per-coefficient map (Eq. 22-24) of one chunk's kept coefficients: the
// mask's set bits are listed in raster order in shared memory, so the threads
// take consecutive output columns and each of the 14 rows is written in whole
// lines.  Nothing is written when the total exceeds the capacity.
__global__ void __launch_bounds__(kMarkThreads) k_map(const float *__restrict__ A, int64_t chan, int nx, int ny,
                                                      const __grid_constant__ BandTab t,
                                                      const uint32_t *__restrict__ mask,
                                                      const uint32_t *__restrict__ count,
                                                      const int64_t *__restrict__ first,
                                                      const int64_t *__restrict__ total,
                                                      const MapTab *__restrict__ tab, float *__restrict__ P,
                                                      int64_t stride)
{
    static_assert(kChunk / 32 == kMarkThreads && kChunk <= 65536, "one mask word per thread, 16-bit positions");
    __shared__ uint16_t list[kChunk];
    __shared__ uint32_t warp_sum[kMarkThreads / 32];
    const uint32_t kept = count[blockIdx.x];
    if (kept == 0 || *total > stride) return;             // block-uniform
    const int tid = threadIdx.x;
    const int b = band_of(t.chunk0, t.nb, blockIdx.x);
    const int64_t i0 = (int64_t)(blockIdx.x - t.chunk0[b]) * kChunk;
    uint32_t word = i0 + tid * 32 < t.n[b] ? mask[(t.voff[b] + i0) / 32 + tid] : 0u, all;
    uint32_t at = block_scan<kMarkThreads>(__popc(word), warp_sum, all);
    for (; word; word &= word - 1) list[at++] = (uint16_t)(tid * 32 + __ffs(word) - 1);
    __syncthreads();
    const MapEntry me = tab->e[b];
    const int64_t out = first[blockIdx.x];
    for (uint32_t k = tid; k < kept; k += kMarkThreads) {
        const int64_t pos = out + k;
        int x, y, z;
        const int64_t e = pyramid_index(t, b, i0 + list[k], nx, ny, x, y, z);
        float amp[4];
        for (int c = 0; c < 4; c++) amp[c] = me.s * fabsf(A[c * chan + e]) * me.w;
        const float step = (float)(1 << me.j);
        P[0 * stride + pos] = me.u[0] + step * x + 0.5f;
        P[1 * stride + pos] = me.u[1] + step * y + 0.5f;
        P[2 * stride + pos] = me.u[2] + step * z + 0.5f;
        for (int d = 0; d < 3; d++) P[(3 + d) * stride + pos] = me.log_scale[d];
        for (int d = 0; d < 4; d++) P[(6 + d) * stride + pos] = me.quat[d];
        // floor 2/255: a retained coefficient stays above the 1/255 cut-off
        const float op = fminf(fmaxf(amp[3], 2.f / 255.f), 0.99f);
        P[10 * stride + pos] = logf(op / (1.f - op));
        P[11 * stride + pos] = amp[0];
        P[12 * stride + pos] = amp[1];
        P[13 * stride + pos] = amp[2];
    }
}

// ------------------------------------------------------------- helpers

std::vector<Band> bands_of(const int dims[3], int levels)
{
    std::vector<Band> out;
    for (int j = 1; j <= levels; j++)
        for (int code = 0; code < 8; code++) {
            if (code == 0 && j != levels) continue;
            Band b;
            b.j = j;
            b.o[0] = code & 1; b.o[1] = (code >> 1) & 1; b.o[2] = (code >> 2) & 1;
            b.mx = dims[0] >> j; b.my = dims[1] >> j; b.mz = dims[2] >> j;
            b.ox = b.o[0] * b.mx; b.oy = b.o[1] * b.my; b.oz = b.o[2] * b.mz;
            b.n = (int64_t)b.mx * b.my * b.mz;
            out.push_back(b);
        }
    return out;
}

// Element offsets, marking chunks and selection blocks of the bands.  Bands of
// at most kSmallBand elements have no blocks in the selection passes (a block of
// the first launch runs all passes of one); of the others a block takes at least
// 8192 elements, and beyond that the blocks are two to an SM, shared out by band
// size.
BandTab band_table(const std::vector<Band> &bands, double beta_N)
{
    BandTab t{};
    t.nb = (int)bands.size();
    int64_t all = 0, off = 0;
    for (const Band &B : bands) all += B.n;
    const int64_t per = std::max<int64_t>(8192, all / (2 * (int64_t)num_sms()) + 1);
    for (int b = 0; b < t.nb; b++) {
        const Band &B = bands[b];
        t.ox[b] = B.ox; t.oy[b] = B.oy; t.oz[b] = B.oz; t.mx[b] = B.mx; t.my[b] = B.my;
        t.n[b] = B.n;
        t.n_beta[b] = std::pow((double)B.n, beta_N);
        t.voff[b] = off;
        off += (B.n + 31) / 32 * 32;
        t.chunk0[b + 1] = t.chunk0[b] + (int)((B.n + kChunk - 1) / kChunk);
        t.blk0[b + 1] = t.blk0[b] + (B.n <= kSmallBand ? 0 : (int)((B.n + per - 1) / per));
    }
    return t;
}

// Device scratch of one build, in order; with ws = NULL only its size.
struct BuildScratch {
    float *A, *tmp, *v;
    uint32_t *mask, *count;
    int64_t *first;
    MapTab *map;
    char *zeroed;            // from here on cleared at the start of a build
    SubState *st;
    double *E;
    uint32_t *hist, *ticket;
    int64_t *total;
    size_t bytes, zero_bytes;
};

BuildScratch build_scratch(void *ws, const int dims[3])
{
    const size_t n = (size_t)dims[0] * dims[1] * dims[2], padded = n + 32 * kMaxBands;
    BuildScratch s{};
    size_t at = (256 - (reinterpret_cast<uintptr_t>(ws) & 255)) & 255;     // 256-byte aligned whatever ws is
    auto take = [&](size_t bytes) {
        char *p = reinterpret_cast<char *>(ws) + at;
        at += (bytes + 255) / 256 * 256;
        return p;
    };
    const size_t chunks = n / kChunk + kMaxBands;
    s.A = (float *)take(4 * n * sizeof(float));                            // RF / pyramid
    s.tmp = (float *)take((size_t)pyramid_tmp_floats(dims) * sizeof(float));   // DWT temporaries
    s.v = (float *)take(padded * sizeof(float));                           // joint magnitudes
    s.mask = (uint32_t *)take(padded / 32 * sizeof(uint32_t));
    s.count = (uint32_t *)take(chunks * sizeof(uint32_t));
    s.first = (int64_t *)take(chunks * sizeof(int64_t));
    s.map = (MapTab *)take(sizeof(MapTab));
    const size_t z0 = at;
    s.zeroed = reinterpret_cast<char *>(ws) + at;
    s.st = (SubState *)take(kMaxBands * sizeof(SubState));
    s.E = (double *)take(kMaxBands * sizeof(double));
    s.ticket = (uint32_t *)take(sizeof(uint32_t));
    s.total = (int64_t *)take(sizeof(int64_t));
    s.hist = (uint32_t *)take((size_t)kMaxBands * kTargets * kBins * sizeof(uint32_t));
    s.zero_bytes = at - z0;
    s.bytes = at + 256;                                                    // room to align the next ws
    return s;
}

vbm_status check_tf(const vbm_tf *tf)
{
    VBM_ARG(tf->n_knots >= 2 && tf->n_knots <= 16, "n_knots must be in [2, 16]");
    for (int i = 1; i < tf->n_knots; i++) VBM_ARG(tf->x[i] > tf->x[i - 1], "TF knots must be ascending");
    return VBM_OK;
}

}  // namespace

size_t build_workspace_bytes(const int dims[3], int levels)
{
    (void)levels;
    return build_scratch(nullptr, dims).bytes;
}

}  // namespace vbm

using namespace vbm;

extern "C" {

vbm_status vbm_tf_apply(const float *d_volume, int64_t n, const vbm_tf *tf, float *d_rf, void *stream)
{
    VBM_ARG(d_volume && tf && d_rf && n >= 0, "invalid argument");
    vbm_status s = check_tf(tf);
    if (s != VBM_OK || n == 0) return s;
    return tf_apply(d_volume, n, tf, d_rf, (cudaStream_t)stream);
}

vbm_status vbm_dwt3d(float *d_data, int n_channels, const int dims[3], int levels, int wavelet, float *d_tmp,
                     void *stream)
{
    VBM_ARG(d_data && dims && d_tmp && n_channels >= 1, "invalid argument");
    VBM_ARG(levels >= 1 && levels <= 9, "levels must be in [1, 9]");
    VBM_ARG(wavelet == 0 || wavelet == 1, "wavelet must be 0 or 1");
    for (int d = 0; d < 3; d++)
        VBM_ARG(dims[d] > 0 && dims[d] % (1 << levels) == 0, "dims must be divisible by 2^levels");
    return dwt_channels(d_data, n_channels, dims, levels, wavelet, d_tmp, (cudaStream_t)stream);
}

vbm_status vbm_build_workspace_size(const int dims[3], int levels, size_t *bytes)
{
    VBM_ARG(dims && bytes, "null argument");
    *bytes = build_workspace_bytes(dims, levels);
    return VBM_OK;
}

vbm_status vbm_build(const float *d_volume, const int dims[3], const vbm_tf *tf, const vbm_bank *bank,
                     const vbm_select *sel, float *d_params, int64_t capacity, int64_t *n_out, float *d_coef,
                     uint8_t *d_keep, void *d_ws, size_t ws_bytes, void *stream)
{
    VBM_ARG(d_volume && dims && tf && bank && sel && n_out && d_ws, "null argument");
    VBM_ARG(capacity >= 0 && (capacity == 0 || d_params), "invalid params buffer");
    const int levels = bank->levels;
    VBM_ARG(levels >= 1 && levels <= 9 && bank->n_sub == 7 * levels + 1, "invalid bank");
    for (int d = 0; d < 3; d++)
        VBM_ARG(dims[d] > 0 && dims[d] % (1 << levels) == 0, "dims must be divisible by 2^levels");
    VBM_ARG(ws_bytes >= build_workspace_bytes(dims, levels), "build workspace too small");
    VBM_ARG(sel->K_tot > 0 && sel->min_per_band >= 0, "invalid selection parameters");
    vbm_status s = check_tf(tf);
    if (s != VBM_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t n = (int64_t)dims[0] * dims[1] * dims[2];
    const BuildScratch w = build_scratch(d_ws, dims);
    float *A = w.A, *v = w.v;
    std::vector<Band> bands = bands_of(dims, levels);
    const int nb = (int)bands.size();
    MapTab map{};
    for (int b = 0; b < nb; b++) {
        const Band &B = bands[b];
        const vbm_bank_entry &e = bank->sub[b];
        VBM_ARG(e.j == B.j && e.o[0] == B.o[0] && e.o[1] == B.o[1] && e.o[2] == B.o[2], "bank order mismatch");
        MapEntry &me = map.e[b];
        for (int d = 0; d < 3; d++) {
            me.u[d] = (float)e.u[d];
            me.log_scale[d] = e.log_scale[d];
        }
        for (int d = 0; d < 4; d++) me.quat[d] = e.quat[d];
        me.w = (float)e.w;
        me.j = B.j;
        me.s = sel->energy_comp ? (float)std::pow(2.0, -1.5 * B.j) : 1.f;
    }
    const BandTab t = band_table(bands, sel->beta_N);
    const Budget bud{sel->alpha_E, (double)sel->K_tot, sel->min_per_band, (float)sel->lambda_mad};

    VBM_CUDA(cudaMemcpyAsync(w.map, &map, sizeof(map), cudaMemcpyHostToDevice, st));
    VBM_CUDA(cudaMemsetAsync(w.zeroed, 0, w.zero_bytes, st));
    s = pyramid_from_volume(d_volume, dims, tf, levels, bank->wavelet, A, w.tmp, v, t.voff, w.E, st);
    if (s != VBM_OK) return s;
    const int chunks = t.chunk0[nb], blocks = t.blk0[nb];
    // the first pass's last nb blocks do all of the small bands' selection
    k_select_pass<0, false><<<blocks + nb, kSelThreads, 0, st>>>(v, t, bud, w.E, w.st, w.hist);
    if (blocks > 0) {
        k_select_pass<1, false><<<blocks, kSelThreads, 0, st>>>(v, t, bud, w.E, w.st, w.hist);
        k_select_pass<2, false><<<blocks, kSelThreads, 0, st>>>(v, t, bud, w.E, w.st, w.hist);
        k_select_pass<0, true><<<blocks, kSelThreads, 0, st>>>(v, t, bud, w.E, w.st, w.hist);
        k_select_pass<1, true><<<blocks, kSelThreads, 0, st>>>(v, t, bud, w.E, w.st, w.hist);
        k_select_pass<2, true><<<blocks, kSelThreads, 0, st>>>(v, t, bud, w.E, w.st, w.hist);
    }
    VBM_LAUNCH("select");
    k_mark<<<chunks, kMarkThreads, 0, st>>>(v, t, dims[0], dims[1], w.st, w.mask, w.count, w.first, w.total, w.ticket,
                                            d_keep);
    VBM_LAUNCH("mark");
    int64_t total = 0;
    VBM_CUDA(cudaMemcpyAsync(&total, w.total, sizeof(total), cudaMemcpyDeviceToHost, st));
    if (capacity > 0) {
        k_map<<<chunks, kMarkThreads, 0, st>>>(A, n, dims[0], dims[1], t, w.mask, w.count, w.first, w.total, w.map,
                                               d_params, capacity);
        VBM_LAUNCH("map");
    }
    if (d_coef) VBM_CUDA(cudaMemcpyAsync(d_coef, A, 4 * n * sizeof(float), cudaMemcpyDeviceToDevice, st));
    VBM_CUDA(cudaStreamSynchronize(st));
    *n_out = total;
    if (total > capacity) {
        set_error("vbm_build: " + std::to_string(total) + " Gaussians kept, capacity " + std::to_string(capacity));
        return VBM_ERR_CAPACITY;
    }
    return VBM_OK;
}

}  // extern "C"
