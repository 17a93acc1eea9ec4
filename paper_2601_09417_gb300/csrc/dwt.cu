// Transfer function and periodised separable 3D wavelet transform (Sec. 3,
// Eq. 1-3; Sec. 4.3, Eq. 20-21) in the Mallat layout.
//
// One level is two kernels: k_dwt_xy transforms along x and y, plane by plane,
// and k_dwt_z along z.  Every filter is a chain of fused multiply-adds in the
// order of its taps, along x, then y, then z, so how the work is split does
// not change a bit of the result.
//
// Traffic of a level: each plane is read once and written once by either
// kernel; vbm_build's first level reads the scalar volume itself and applies
// the transfer function where the rows are staged, so the four RGBA channels
// are never stored untransformed.  Against one gather kernel an axis (a 64-bit
// division and a modulo for every tap, three reads and writes of each value):
// tf_apply + four-level dwt3d of 4 x 256^3, 4.30 -> 0.32 ms; vbm_build of a
// 512^3 volume, 36.3 -> 3.9 ms.
#include "tf_dev.h"

namespace vbm {

namespace {

// Filter taps, low-pass then high-pass, passed by value: calls on different
// streams or with different wavelets share nothing.
struct Taps {
    float lo[9], hi[9];
};

// Tap ranges relative to the even sample 2k: a[k] sums x[2k + LO], ..., and
// d[k] sums x[2k + HI], ...; PAIRS sample pairs from 2k + FIRST on cover both.
template <int WAVELET>
struct Wavelet;
template <>
struct Wavelet<0> {     // bior4.4: 9 and 7 taps
    static constexpr int LO = -4, LO_LEN = 9, HI = -2, HI_LEN = 7, FIRST = -4, PAIRS = 5;
};
template <>
struct Wavelet<1> {     // Haar
    static constexpr int LO = 0, LO_LEN = 2, HI = 0, HI_LEN = 2, FIRST = 0, PAIRS = 1;
};

Taps make_taps(int wavelet)
{
    const FilterBank fb = make_filters(wavelet);
    Taps t{};
    int k = 0;
    for (auto &kv : fb.ht) t.lo[k++] = (float)kv.second;
    k = 0;
    for (auto &kv : fb.gt) t.hi[k++] = (float)kv.second;
    return t;
}

__device__ __forceinline__ int wrap(int i, int n)
{
    i %= n;
    return i < 0 ? i + n : i;
}

constexpr int kXYThreads = 128;
constexpr int kXPer = 4;                 // x positions (two output pairs) a thread
constexpr int kMaxSlot = 32;             // threads of a slot: 128 positions
constexpr int kMinSlot = 8;

// Where the rows of the x and y passes come from: an array read one value or
// (rows of whole, aligned 16-byte words) four values at a time, or the scalar
// volume through the transfer function.
enum Source { kScalar, kQuads, kTransfer };

// x and y passes.  A slot of `1 << slot_log` threads takes one strip: a tile
// of 4 x positions a thread, `pairs` row pairs, one plane, one channel.  Rows
// enter in order, two at a time: staged in shared memory (double-buffered, the
// next two rows in flight in registers), filtered along x (each thread reads
// its 12 inputs as three 16-byte words for four outputs) and kept in a
// register ring of the 10 rows the y filter spans, from which every new row
// pair gives one low and one high output row.  A row is therefore read once a
// strip (plus the 8 rows of overlap between strips), not once a tap, and
// nothing goes to memory between the two passes.  The y filter takes a
// thread's columns in pairs (FP32x2) and rows of whole 16-byte words are
// staged four values at a time: the kernel is bound by instruction issue, not
// by the arithmetic itself (4 x 256^3, all levels: 200 -> 170 us; with the
// transfer function on 512^3, first level: 2.76 -> 1.63 ms).  A slot lies in
// one warp, so that only the transfer function's four need a block barrier
// (with slots of 64 threads and barriers for all the 4 x 256^3 pyramid took 395
// us instead of 367, before the z pass's asynchronous copies below).
//
// kTransfer: the source is the scalar volume; four neighbouring slots take the
// four channels of one strip, whose threads share the loads and the transfer
// function's evaluation (the two rows' positions in one sequence, so that the
// 16 beyond the threads cost one warp one more evaluation, not two).
struct XYArgs {
    const float *src;
    int64_t src_chan, src_plane;         // strides of a channel and a plane
    int src_row;
    float *dst;                          // [channel][plane][sy][sx]
    int64_t dst_chan;
    int sx, sy, sz;                      // region
    int z_first, planes;                 // plane t of dst holds z = (z_first + t) mod sz
    int pairs;                           // row pairs a strip
    int x_tiles, strips_y, slot_log;
    int vec2;                            // low and high rows start on 8-byte boundaries
};

template <int WAVELET, int SOURCE>
__global__ void __launch_bounds__(kXYThreads, 5) k_dwt_xy(const __grid_constant__ XYArgs a,
                                                          const __grid_constant__ Taps w,
                                                          const __grid_constant__ TFDev tf)
{
    using Wv = Wavelet<WAVELET>;
    constexpr int HALO = 4;                                      // staged positions before the tile
    constexpr int R = Wv::PAIRS;
    constexpr int MAX_ROW = kXYThreads * kXPer + 8 * (kXYThreads / kMinSlot);
    constexpr bool TF = SOURCE == kTransfer;
    __shared__ __align__(16) float rows[2][2][MAX_ROW];          // [buffer][row][slot][position]
    __shared__ TFTable table;
    const int slot_threads = 1 << a.slot_log;
    const int tile = slot_threads * kXPer, width = tile + 8;     // staged positions of a row
    const int slot = threadIdx.x >> a.slot_log, p = threadIdx.x & (slot_threads - 1);
    const int slots = kXYThreads >> a.slot_log;
    // the strip of this slot; with TF four slots share one
    const int64_t strip = TF ? (int64_t)blockIdx.x * (slots / 4) + slot / 4 : (int64_t)blockIdx.x * slots + slot;
    const int chan = TF ? slot & 3 : blockIdx.y;
    const int64_t n_strips = (int64_t)a.x_tiles * a.strips_y * a.planes;
    const bool on = strip < n_strips;
    const int64_t s = on ? strip : 0;
    const int xt = (int)(s % a.x_tiles), yt = (int)((s / a.x_tiles) % a.strips_y), zt = (int)(s / a.x_tiles / a.strips_y);
    const int x0 = xt * tile, k0 = yt * a.pairs;
    const int k1 = on ? min(a.sy / 2, k0 + a.pairs) : k0;        // output row pairs [k0, k1)
    if (TF) tf_stage(tf, table);
    const float *row0 = a.src + (TF ? 0 : chan * a.src_chan) + (int64_t)wrap(a.z_first + zt, a.sz) * a.src_plane;
    int y = wrap(2 * k0 + Wv::FIRST, a.sy);
    const float *row = row0 + (int64_t)y * a.src_row;
    auto next_row = [&]() {
        y++;
        row += a.src_row;
        if (y == a.sy) {
            y = 0;
            row = row0;
        }
    };
    // this thread's part of two rows in flight, and where it goes
    constexpr int LOADS = TF ? 3 : SOURCE == kQuads ? 4 : 2 * (kXPer + 1);
    float raw[SOURCE == kQuads ? 1 : LOADS];
    float4 raw4[SOURCE == kQuads ? LOADS : 1];
    const int loaders = 4 * slot_threads, q = threadIdx.x & (loaders - 1);   // TF: the strip's threads
    int col[LOADS];
#pragma unroll
    for (int i = 0; i < LOADS; i++) {
        if (TF) {
            const int at = q + i * loaders;
            col[i] = wrap(x0 - HALO + (at < width ? at : at - width), a.sx);
        } else if (SOURCE == kQuads) {
            col[i] = wrap(i & 1 ? (p == 0 ? x0 - HALO : x0 + tile) : x0 + 4 * p, a.sx);
        } else {
            col[i] = wrap(x0 - HALO + p + (i >> 1) * slot_threads, a.sx);
        }
    }
    const bool second_is_row1 = q + loaders >= width;            // TF: the row of the second load
    auto fetch = [&]() {
        const float *r0 = row;
        next_row();
        const float *r1 = row;
        next_row();
        if constexpr (TF) {
            raw[0] = r0[col[0]];
            raw[1] = (second_is_row1 ? r1 : r0)[col[1]];
            if (q < 16) raw[2] = r1[col[2]];
        } else if constexpr (SOURCE == kQuads) {
            raw4[0] = *reinterpret_cast<const float4 *>(r0 + col[0]);
            raw4[2] = *reinterpret_cast<const float4 *>(r1 + col[2]);
            if (p < 2) {
                raw4[1] = *reinterpret_cast<const float4 *>(r0 + col[1]);
                raw4[3] = *reinterpret_cast<const float4 *>(r1 + col[3]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < LOADS; i++)
                if (p + (i >> 1) * slot_threads < width) raw[i] = (i & 1 ? r1 : r0)[col[i]];
        }
    };
    auto stage = [&](int buf) {
        if constexpr (TF) {
            // a loop, so that the evaluation is compiled once a step: inlined
            // three times in each of the five unrolled steps it overran the
            // instruction cache
            float *to = &rows[buf][0][(slot & ~3) * width];
            float v = raw[0];
            const int count = q < 16 ? 3 : 2;
#pragma unroll 1
            for (int i = 0; i < count; i++) {
                const float4 c = tf_apply(tf, table, v);
                int at = q + i * loaders;
                at += at < width ? 0 : MAX_ROW - width;          // the second row
                to[at] = c.x;
                to[at + width] = c.y;
                to[at + 2 * width] = c.z;
                to[at + 3 * width] = c.w;
                v = i == 0 ? raw[1] : raw[2];
            }
        } else if constexpr (SOURCE == kQuads) {
            float *to = &rows[buf][0][slot * width];
            *reinterpret_cast<float4 *>(to + HALO + 4 * p) = raw4[0];
            *reinterpret_cast<float4 *>(to + MAX_ROW + HALO + 4 * p) = raw4[2];
            if (p < 2) {
                const int at = p == 0 ? 0 : HALO + tile;
                *reinterpret_cast<float4 *>(to + at) = raw4[1];
                *reinterpret_cast<float4 *>(to + MAX_ROW + at) = raw4[3];
            }
        } else {
#pragma unroll
            for (int i = 0; i < LOADS; i++) {
                const int at = p + (i >> 1) * slot_threads;
                if (at < width) rows[buf][i & 1][slot * width + at] = raw[i];
            }
        }
    };
    const int hx = a.sx >> 1, hy = a.sy >> 1;
    const int xo = x0 / 2 + 2 * p;                               // low column of the first pair
    float *dst = a.dst + chan * a.dst_chan + (int64_t)zt * a.sx * a.sy + xo;
    const int64_t high_rows = (int64_t)hy * a.sx;
    const bool two = a.vec2 && xo + 1 < hx;                      // both pairs exist and can be stored as one
    float2 ring[R][2][2];                                        // x results: low pair, high pair
    auto x_filter = [&](int buf, float2 (&out)[2][2]) {
#pragma unroll
        for (int r = 0; r < 2; r++) {
            const float4 *in4 = reinterpret_cast<const float4 *>(&rows[buf][r][slot * width + kXPer * p]);
            const float4 A = in4[0], B = in4[1], C = in4[2];
            const float in[12] = {A.x, A.y, A.z, A.w, B.x, B.y, B.z, B.w, C.x, C.y, C.z, C.w};
            float lo[2], hi[2];
#pragma unroll
            for (int k = 0; k < 2; k++) {
                lo[k] = hi[k] = 0.f;
#pragma unroll
                for (int t = 0; t < Wv::LO_LEN; t++) lo[k] = __fmaf_rn(w.lo[t], in[HALO + 2 * k + Wv::LO + t], lo[k]);
#pragma unroll
                for (int t = 0; t < Wv::HI_LEN; t++) hi[k] = __fmaf_rn(w.hi[t], in[HALO + 2 * k + Wv::HI + t], hi[k]);
            }
            out[r][0] = make_float2(lo[0], lo[1]);
            out[r][1] = make_float2(hi[0], hi[1]);
        }
    };
    auto put = [&](float *d, float2 v) {                         // two neighbouring outputs
        if (two) {
            *reinterpret_cast<float2 *>(d) = v;
        } else {
            if (xo < hx) d[0] = v.x;
            if (xo + 1 < hx) d[1] = v.y;
        }
    };
    const int steps = a.pairs + R - 1;                           // the same for every slot of the block
    float *out = dst + (int64_t)k0 * a.sx;
    fetch();
    __syncthreads();                                             // the table
    for (int s0 = 0; s0 < steps; s0 += R) {
#pragma unroll
        for (int u = 0; u < R; u++) {                            // ring positions are compile-time
            const int step = s0 + u;
            if (step >= steps) break;
            stage(step & 1);
            if (step + 1 < steps) fetch();
            if (TF) __syncthreads();
            else __syncwarp();                                   // a slot lies in one warp
            x_filter(step & 1, ring[u]);
            if (step < R - 1 || k0 + step - (R - 1) >= k1) continue;
            // sample pair i of the window is ring slot (u + 1 + i) mod R
            float2 lo[2], hi[2];
            lo[0] = lo[1] = hi[0] = hi[1] = make_float2(0.f, 0.f);
#pragma unroll
            for (int t = 0; t < Wv::LO_LEN; t++) {
                const int i = Wv::LO - Wv::FIRST + t;
#pragma unroll
                for (int c = 0; c < 2; c++)
                    lo[c] = __ffma2_rn(make_float2(w.lo[t], w.lo[t]), ring[(u + 1 + i / 2) % R][i & 1][c], lo[c]);
            }
#pragma unroll
            for (int t = 0; t < Wv::HI_LEN; t++) {
                const int i = Wv::HI - Wv::FIRST + t;
#pragma unroll
                for (int c = 0; c < 2; c++)
                    hi[c] = __ffma2_rn(make_float2(w.hi[t], w.hi[t]), ring[(u + 1 + i / 2) % R][i & 1][c], hi[c]);
            }
            put(out, lo[0]);
            put(out + hx, lo[1]);
            put(out + high_rows, hi[0]);
            put(out + high_rows + hx, hi[1]);
            out += a.sx;
        }
    }
}

// z pass: a thread takes V neighbouring columns of NC channels and `pairs`
// plane pairs, with the 10 planes the filter spans in a register ring and the
// next pairs' loads in flight.  Bound by memory: each value is read and
// written once (plus the 8 planes of overlap between chunks, from L2).
struct ZArgs {
    const float *src;                    // [channel][plane][sy][sx]
    int64_t src_chan;
    int planes, z_first;                 // plane t holds z = z_first + t (modulo planes)
    float *dst;                          // Mallat layout, strides below
    int64_t dst_chan, dst_plane;
    int dst_row;
    int sx, sy, sz;
    int k_begin, k_end, pairs;           // output pairs of this launch, and of a thread
};

// What vbm_build selects by, written where the level's coefficients are formed
// (NC = 4, V = 1): the joint magnitude of each, at its place in its subband,
// and the subband's opacity energy.  Octant c = o_x + 2 o_y + 4 o_z is subband
// band[c] (-1: the low octant of a level that is not the last) and its
// magnitudes start at voff[c].  A pass of its own read the four channels again
// (732 us of a 512^3 build; the fused stores and the energies' double
// precision sums add 185 us).
struct Magnitudes {
    float *v;
    double *E;
    int64_t voff[8];
    int band[8];
};

template <int V>
struct Vec;
template <>
struct Vec<1> { using T = float; };
template <>
struct Vec<4> { using T = float4; };

constexpr int kZDepth = 4;               // plane pairs in flight, a power of two

// Asynchronous copies of 4 or 16 bytes into shared memory.
__device__ __forceinline__ void copy_async(float *to, const float *from)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from)
                 : "memory");
}

__device__ __forceinline__ void copy_async(float4 *to, const float *from)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from)
                 : "memory");
}

__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

// At most N of the thread's groups still in flight.
template <int N>
__device__ __forceinline__ void copy_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Threads a block: with four channels a thread takes up to 102 registers, and
// blocks of 128 then leave 20 warps on an SM (of 256: 16).
__host__ __device__ constexpr int z_threads(int channels) { return channels == 4 ? 128 : 256; }

template <int WAVELET, int V, int NC>
__global__ void __launch_bounds__(z_threads(NC), NC == 4 ? 5 : 3) k_dwt_z(const __grid_constant__ ZArgs a, const __grid_constant__ Taps w,
                                                     const __grid_constant__ Magnitudes mag)
{
    using Wv = Wavelet<WAVELET>;
    using T = typename Vec<V>::T;
    constexpr int R = Wv::PAIRS;
    constexpr bool MAG = NC == 4;
    constexpr int THREADS = z_threads(NC);
    const int64_t plane = (int64_t)a.sx * a.sy;
    int64_t at = ((int64_t)blockIdx.x * THREADS + threadIdx.x) * V;
    const bool on = at < plane;
    if (!MAG && !on) return;             // with MAG every lane stays for the energies' sum
    if (!on) at = 0;
    const int k0 = a.k_begin + blockIdx.y * a.pairs, k1 = min(a.k_end, k0 + a.pairs);
    const int y = (int)(at / a.sx), x = (int)(at - (int64_t)y * a.sx);
    const float *src = a.src + blockIdx.z * a.src_chan + at;
    float *dst = a.dst + blockIdx.z * a.dst_chan + (int64_t)y * a.dst_row + x;
    const int hx = a.sx >> 1, hy = a.sy >> 1;
    const int code = (x >= hx) + 2 * (y >= hy);                  // MAG: octants code and code + 4
    float *v_lo = nullptr, *v_hi = nullptr;
    double e_lo = 0.0, e_hi = 0.0;
    if (MAG && on) {
        const int64_t in_plane = (int64_t)(y - (y >= hy ? hy : 0)) * hx + (x - (x >= hx ? hx : 0));
        if (mag.band[code] >= 0) v_lo = mag.v + mag.voff[code] + in_plane;
        v_hi = mag.v + mag.voff[code + 4] + in_plane;
    }
    // plane pairs on their way: copied asynchronously into the thread's own
    // shared-memory words, so that the depth costs no registers (one pair ahead
    // in registers left too few bytes in flight: 4 x 256^3 pyramid 395 -> 354
    // us, with the slots within a warp above 327; vbm_build of 512^3 4.27 -> 4.07
    // ms)
    __shared__ T stage[kZDepth][2][NC][THREADS];
    int t = wrap(2 * k0 + Wv::FIRST - a.z_first, a.planes);
    float ring[R][2][NC * V];
    auto fetch = [&](int slot) {
#pragma unroll
        for (int r = 0; r < 2; r++) {
#pragma unroll
            for (int n = 0; n < NC; n++)
                copy_async(&stage[slot][r][n][threadIdx.x], src + n * a.src_chan + (int64_t)t * plane);
            t = t + 1 == a.planes ? 0 : t + 1;
        }
    };
    // sqrt(((a0 a0 + a1 a1) + a2 a2) + a3 a3), rounded op by op
    auto magnitude = [](const float *c) {
        float acc = __fmul_rn(c[0], c[0]);
        acc = __fadd_rn(acc, __fmul_rn(c[1], c[1]));
        acc = __fadd_rn(acc, __fmul_rn(c[2], c[2]));
        return __fsqrt_rn(__fadd_rn(acc, __fmul_rn(c[3], c[3])));
    };
    const int steps = k1 - k0 + R - 1;
#pragma unroll
    for (int s = 0; s < kZDepth - 1; s++) {
        if (s < steps) fetch(s);
        copy_commit();
    }
    for (int s0 = 0; s0 < steps; s0 += R) {
#pragma unroll
        for (int u = 0; u < R; u++) {
            const int step = s0 + u;
            if (step >= steps) break;
            if (step + kZDepth - 1 < steps) fetch((step + kZDepth - 1) % kZDepth);
            copy_commit();
            copy_wait<kZDepth - 1>();
#pragma unroll
            for (int r = 0; r < 2; r++)
#pragma unroll
                for (int n = 0; n < NC; n++)
                    *reinterpret_cast<T *>(&ring[u][r][n * V]) = stage[step % kZDepth][r][n][threadIdx.x];
            if (step < R - 1) continue;
            const int k = k0 + step - (R - 1);
            float lo[NC * V], hi[NC * V];
#pragma unroll
            for (int c = 0; c < NC * V; c++) lo[c] = hi[c] = 0.f;
#pragma unroll
            for (int i = 0; i < Wv::LO_LEN; i++) {
                const int j = Wv::LO - Wv::FIRST + i;
#pragma unroll
                for (int c = 0; c < NC * V; c++)
                    lo[c] = __fmaf_rn(w.lo[i], ring[(u + 1 + j / 2) % R][j & 1][c], lo[c]);
            }
#pragma unroll
            for (int i = 0; i < Wv::HI_LEN; i++) {
                const int j = Wv::HI - Wv::FIRST + i;
#pragma unroll
                for (int c = 0; c < NC * V; c++)
                    hi[c] = __fmaf_rn(w.hi[i], ring[(u + 1 + j / 2) % R][j & 1][c], hi[c]);
            }
            if (MAG && !on) continue;
            float *d_lo = dst + (int64_t)k * a.dst_plane, *d_hi = dst + (int64_t)(a.sz / 2 + k) * a.dst_plane;
#pragma unroll
            for (int n = 0; n < NC; n++) {
                *reinterpret_cast<T *>(d_lo + n * a.dst_chan) = *reinterpret_cast<const T *>(&lo[n * V]);
                *reinterpret_cast<T *>(d_hi + n * a.dst_chan) = *reinterpret_cast<const T *>(&hi[n * V]);
            }
            if constexpr (MAG) {
                const int64_t in_band = (int64_t)k * hx * hy;
                if (v_lo) {
                    v_lo[in_band] = magnitude(lo);
                    e_lo += (double)lo[3] * (double)lo[3];
                }
                v_hi[in_band] = magnitude(hi);
                e_hi += (double)hi[3] * (double)hi[3];
            }
        }
    }
    if constexpr (MAG) {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int c = 0; c < 4; c++) {
            if (!__any_sync(0xffffffffu, on && code == c)) continue;
            double lo = on && code == c ? e_lo : 0.0, hi = on && code == c ? e_hi : 0.0;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                lo += __shfl_xor_sync(0xffffffffu, lo, off);
                hi += __shfl_xor_sync(0xffffffffu, hi, off);
            }
            if (lane == 0) {
                if (mag.band[c] >= 0) atomicAdd(mag.E + mag.band[c], lo);
                atomicAdd(mag.E + mag.band[c + 4], hi);
            }
        }
    }
}

constexpr int kTFThreads = 256;

// d_rf = TF(volume): four elements a thread where both arrays allow 16-byte
// accesses (VEC), one otherwise.
template <bool VEC>
__global__ void __launch_bounds__(kTFThreads) k_tf_apply(const float *__restrict__ F, int64_t n,
                                                         const __grid_constant__ TFDev tf, float *__restrict__ RF)
{
    __shared__ TFTable table;
    tf_stage(tf, table);
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * kTFThreads + threadIdx.x;
    if constexpr (VEC) {
        if (4 * i >= n) return;
        const float4 f = reinterpret_cast<const float4 *>(F)[i];
        const float4 a = tf_apply(tf, table, f.x), b = tf_apply(tf, table, f.y), c = tf_apply(tf, table, f.z),
                     d = tf_apply(tf, table, f.w);
        float4 *out = reinterpret_cast<float4 *>(RF) + i;
        const int64_t step = n / 4;
        out[0] = make_float4(a.x, b.x, c.x, d.x);
        out[step] = make_float4(a.y, b.y, c.y, d.y);
        out[2 * step] = make_float4(a.z, b.z, c.z, d.z);
        out[3 * step] = make_float4(a.w, b.w, c.w, d.w);
    } else {
        if (i >= n) return;
        const float4 a = tf_apply(tf, table, F[i]);
        RF[i] = a.x;
        RF[n + i] = a.y;
        RF[2 * n + i] = a.z;
        RF[3 * n + i] = a.w;
    }
}

bool aligned(const void *p, size_t to) { return reinterpret_cast<uintptr_t>(p) % to == 0; }

// Work a strip (row pairs) or a z chunk (plane pairs): the longest, up to
// `most`, that still leaves `units` threads' worth of parallel work four waves
// of the chip; the 8 rows or planes of overlap cost 8 / (2 pairs).
int pairs_per(int total_pairs, int64_t lanes, int most)
{
    int per = std::min(most, total_pairs);
    const int64_t want = (int64_t)num_sms() * 1024;
    while (per > 4 && lanes * ((total_pairs + per - 1) / per) < want) per = (per + 1) / 2;
    return std::max(per, 1);
}

template <int WAVELET, bool TF>
vbm_status launch_xy(XYArgs a, int channels, const Taps &w, const TFDev &tf, cudaStream_t st)
{
    int log = 3;
    while ((1 << log) * kXPer < a.sx && (1 << log) < kMaxSlot) log++;
    a.slot_log = log;
    const int tile = (1 << log) * kXPer;
    a.x_tiles = (a.sx + tile - 1) / tile;
    a.pairs = pairs_per(a.sy / 2, ((int64_t)a.x_tiles * a.planes * channels) << log, 32);
    a.strips_y = (a.sy / 2 + a.pairs - 1) / a.pairs;
    a.vec2 = aligned(a.dst, 8) && (a.sx / 2) % 2 == 0 && a.dst_chan % 2 == 0;
    const int64_t strips = (int64_t)a.x_tiles * a.strips_y * a.planes;
    const int per_block = (kXYThreads >> log) / (TF ? 4 : 1);
    dim3 grid((unsigned)((strips + per_block - 1) / per_block), TF ? 1 : channels);
    // whole 16-byte words: the region's rows wrap at a multiple of four values
    // and every row starts on a 16-byte boundary
    const bool quads = a.sx % 4 == 0 && aligned(a.src, 16) && a.src_row % 4 == 0 && a.src_plane % 4 == 0 &&
                       a.src_chan % 4 == 0;
    auto kernel = TF ? k_dwt_xy<WAVELET, kTransfer> : quads ? k_dwt_xy<WAVELET, kQuads> : k_dwt_xy<WAVELET, kScalar>;
    kernel<<<grid, kXYThreads, 0, st>>>(a, w, tf);
    VBM_LAUNCH("dwt_xy");
    return VBM_OK;
}

// mag: the magnitudes of a level of four channels (NULL: none).
template <int WAVELET>
vbm_status launch_z(ZArgs a, int channels, const Taps &w, const Magnitudes *mag, cudaStream_t st)
{
    const int64_t plane = (int64_t)a.sx * a.sy;
    const bool vec = !mag && a.sx % 4 == 0 && aligned(a.src, 16) && aligned(a.dst, 16) && a.src_chan % 4 == 0 &&
                     a.dst_chan % 4 == 0 && a.dst_plane % 4 == 0 && a.dst_row % 4 == 0;
    const int64_t lanes = vec ? plane / 4 : plane;
    const int split = mag ? 1 : channels;                        // channels of different threads
    // a grid's second axis holds 65535 chunks: a volume long beyond that in z
    // takes longer ones
    a.pairs = std::max(pairs_per(a.k_end - a.k_begin, lanes * split, 64), (a.k_end - a.k_begin + 65534) / 65535);
    const int threads = z_threads(mag ? 4 : 1);
    dim3 grid((unsigned)((lanes + threads - 1) / threads),
              (unsigned)((a.k_end - a.k_begin + a.pairs - 1) / a.pairs), (unsigned)split);
    if (mag) k_dwt_z<WAVELET, 1, 4><<<grid, threads, 0, st>>>(a, w, *mag);
    else if (vec) k_dwt_z<WAVELET, 4, 1><<<grid, threads, 0, st>>>(a, w, Magnitudes{});
    else k_dwt_z<WAVELET, 1, 1><<<grid, threads, 0, st>>>(a, w, Magnitudes{});
    VBM_LAUNCH("dwt_z");
    return VBM_OK;
}

// One level in place on the region of `channels` channels of data; tmp holds
// them.
template <int WAVELET>
vbm_status dwt_level(float *data, int channels, const int dims[3], int level, float *tmp, const Taps &w,
                     const Magnitudes *mag, cudaStream_t st)
{
    const int64_t n = (int64_t)dims[0] * dims[1] * dims[2], plane = (int64_t)dims[0] * dims[1];
    const int sx = dims[0] >> (level - 1), sy = dims[1] >> (level - 1), sz = dims[2] >> (level - 1);
    XYArgs a{};
    a.src = data;
    a.src_chan = n;
    a.src_plane = plane;
    a.src_row = dims[0];
    a.dst = tmp;
    a.dst_chan = (int64_t)sx * sy * sz;
    a.sx = sx; a.sy = sy; a.sz = sz;
    a.planes = sz;
    vbm_status s = launch_xy<WAVELET, false>(a, channels, w, TFDev{}, st);
    if (s != VBM_OK) return s;
    ZArgs z{};
    z.src = tmp;
    z.src_chan = a.dst_chan;
    z.planes = sz;
    z.dst = data;
    z.dst_chan = n;
    z.dst_plane = plane;
    z.dst_row = dims[0];
    z.sx = sx; z.sy = sy; z.sz = sz;
    z.k_end = sz / 2;
    return launch_z<WAVELET>(z, channels, w, mag, st);
}

template <int WAVELET>
vbm_status dwt_levels(float *data, int n_channels, const int dims[3], int levels, float *tmp, int64_t tmp_floats,
                      const Taps &w, cudaStream_t st)
{
    const int64_t n = (int64_t)dims[0] * dims[1] * dims[2];
    for (int j = 1; j <= levels; j++) {
        const int64_t region = n >> (3 * (j - 1));
        const int most = (int)std::min<int64_t>(n_channels, std::min<int64_t>(tmp_floats / region, 32768));
        for (int c = 0; c < n_channels; c += most) {
            vbm_status s = dwt_level<WAVELET>(data + c * n, std::min(most, n_channels - c), dims, j, tmp, w, nullptr,
                                              st);
            if (s != VBM_OK) return s;
        }
    }
    return VBM_OK;
}

// The RGBA pyramid of a scalar volume with the magnitudes of its subbands.
// The first level reads the volume through the transfer function, in slabs of
// planes where tmp does not hold the four channels whole.
template <int WAVELET>
vbm_status pyramid_levels(const float *volume, const int dims[3], const TFDev &tf, int levels, float *A, float *tmp,
                          int64_t tmp_floats, const Taps &w, float *v, const int64_t *voff, double *E, cudaStream_t st)
{
    using Wv = Wavelet<WAVELET>;
    // the subbands of level j: seven octants, and at the last level the low one first
    auto level_magnitudes = [&](int j) {
        Magnitudes m{v, E, {}, {}};
        for (int c = 0; c < 8; c++) {
            const int b = 7 * (j - 1) + c - (j == levels ? 0 : 1);
            m.band[c] = c == 0 && j != levels ? -1 : b;
            m.voff[c] = m.band[c] < 0 ? 0 : voff[b];
        }
        return m;
    };
    const int64_t plane = (int64_t)dims[0] * dims[1], n = plane * dims[2];
    const int overlap = 2 * (Wv::PAIRS - 1);
    const int64_t room = tmp_floats / (4 * plane);                        // planes of four channels
    const bool whole = room >= dims[2];
    const int slab = whole ? dims[2] / 2 : (int)((room - overlap) / 2);   // output pairs
    const Magnitudes first = level_magnitudes(1);
    for (int k = 0; k < dims[2] / 2; k += slab) {
        const int k1 = std::min(dims[2] / 2, k + slab);
        XYArgs a{};
        a.src = volume;
        a.src_plane = plane;
        a.src_row = dims[0];
        a.dst = tmp;
        a.sx = dims[0]; a.sy = dims[1]; a.sz = dims[2];
        a.z_first = whole ? 0 : 2 * k + Wv::FIRST;
        a.planes = whole ? dims[2] : 2 * (k1 - k) + overlap;
        a.dst_chan = plane * a.planes;
        vbm_status s = launch_xy<WAVELET, true>(a, 4, w, tf, st);
        if (s != VBM_OK) return s;
        ZArgs z{};
        z.src = tmp;
        z.src_chan = a.dst_chan;
        z.planes = a.planes;
        z.z_first = a.z_first;
        z.dst = A;
        z.dst_chan = n;
        z.dst_plane = plane;
        z.dst_row = dims[0];
        z.sx = dims[0]; z.sy = dims[1]; z.sz = dims[2];
        z.k_begin = k;
        z.k_end = k1;
        s = launch_z<WAVELET>(z, 4, w, &first, st);
        if (s != VBM_OK) return s;
    }
    for (int j = 2; j <= levels; j++) {
        const Magnitudes m = level_magnitudes(j);
        vbm_status s = dwt_level<WAVELET>(A, 4, dims, j, tmp, w, &m, st);
        if (s != VBM_OK) return s;
    }
    return VBM_OK;
}

}  // namespace

vbm_status tf_apply(const float *volume, int64_t n, const vbm_tf *tf, float *rf, cudaStream_t st)
{
    const bool vec = n % 4 == 0 && aligned(volume, 16) && aligned(rf, 16);
    const int64_t lanes = vec ? n / 4 : n;
    const unsigned grid = (unsigned)((lanes + kTFThreads - 1) / kTFThreads);
    if (vec) k_tf_apply<true><<<grid, kTFThreads, 0, st>>>(volume, n, to_dev(tf), rf);
    else k_tf_apply<false><<<grid, kTFThreads, 0, st>>>(volume, n, to_dev(tf), rf);
    VBM_LAUNCH("tf_apply");
    return VBM_OK;
}

// tmp: at least 2 nx ny nz floats.
vbm_status dwt_channels(float *data, int n_channels, const int dims[3], int levels, int wavelet, float *tmp,
                        cudaStream_t st)
{
    const int64_t room = 2 * (int64_t)dims[0] * dims[1] * dims[2];
    const Taps w = make_taps(wavelet);
    return wavelet == 1 ? dwt_levels<1>(data, n_channels, dims, levels, tmp, room, w, st)
                        : dwt_levels<0>(data, n_channels, dims, levels, tmp, room, w, st);
}

// Floats of tmp for pyramid_from_volume: the four channels whole up to 2^26
// floats (256^3 volumes), which makes vbm_build's scratch 36 bytes a voxel there
// (604 MB at most); beyond that 1.2 volumes, worked in slabs, and 25 bytes.  Slabs
// of 1.2 volumes throughout would keep 25 bytes everywhere and make vbm_build of
// 128^3 / 224 x 160 x 96 / 256^3 take 336 / 460 / 750 us instead of 291 / 336 /
// 645.  At least half of the volume (the second level's four channels) and 16
// planes.
int64_t pyramid_tmp_floats(const int dims[3])
{
    const int64_t n = (int64_t)dims[0] * dims[1] * dims[2], plane = (int64_t)dims[0] * dims[1];
    const int64_t whole = 4 * n;
    return std::min(whole, std::max({n + n / 5, (int64_t)1 << 26, 4 * plane * 16}));
}

vbm_status pyramid_from_volume(const float *volume, const int dims[3], const vbm_tf *tf, int levels, int wavelet,
                               float *A, float *tmp, float *v, const int64_t *voff, double *E, cudaStream_t st)
{
    const int64_t room = pyramid_tmp_floats(dims);
    const Taps w = make_taps(wavelet);
    const TFDev t = to_dev(tf);
    return wavelet == 1 ? pyramid_levels<1>(volume, dims, t, levels, A, tmp, room, w, v, voff, E, st)
                        : pyramid_levels<0>(volume, dims, t, levels, A, tmp, room, w, v, voff, E, st);
}

}  // namespace vbm
