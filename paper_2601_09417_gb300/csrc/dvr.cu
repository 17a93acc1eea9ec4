// Emission-absorption ray marching of the supervision images (Sec. 4.4:
// "we render 64 images through volumetric integration").
//
// One thread per pixel, warps of 8 x 4 pixels so neighbouring rays sample
// neighbouring voxels (L1/L2 reuse).  Segments of length `step` along the
// clipped ray, sampled at their midpoints with manual trilinear
// interpolation (hardware texture filtering uses 8-bit fractional weights,
// too coarse for 1e-4 images); TF on the interpolated scalar; opacity
// correction a' = 1 - (1 - a)^len; front to back;
// the march stops once T < 1e-6, which changes the result by less than 1e-6.
//
// Empty space.  Where the transfer function has no opacity a sample adds
// nothing, and most of a volume is such space.  With a workspace, k_occupancy
// first marks, one bit a block of 8^3 cells, the blocks that some sample with
// opacity may lie in; a ray then asks once a block, passes an empty one in a
// single step and marches an occupied one without further tests.  Only samples
// whose opacity is 0 are passed over, so the images are those of the full march
// bit for bit.  The marks cost one read of the volume (98 us of 512^3).  Blocks of
// 8^3: with 4^3 a ray asks twice as often for a sixth fewer samples (8 x 1024^2
// of 512^3 8.07 -> 8.83 ms, 8 x 512^2 of 128^3 489 -> 553 us).  All together
// against the full march in 16 x 16 blocks: 21.3 -> 6.0 ms and 1152 -> 410 us.
#include "tf_dev.h"

namespace vbm {
namespace {

constexpr int kCellShift = 3, kCell = 1 << kCellShift;   // cells of a block along each axis
constexpr int kOccupancyCols = 32 * kCell;   // columns of one occupancy word
constexpr int kOccupancyThreads = kOccupancyCols + 32;

// Scalars f <= lo and f >= hi have no opacity: the transfer function's alpha is
// 0 (or less) from its first knot up to a knot at lo, and from a knot at hi to
// its last.  An absent bound is NaN, which no scalar compares with, infinite
// ones included; lo is +infinity where no scalar has opacity.  The margins cover
// the rounding of the interpolated value, so that a block all of whose corners
// lie beyond one of them holds no sample with opacity; with lo = 0 (alpha rises
// from the first knot) corners of at most 0 interpolate to at most 0 exactly.
struct NoOpacity {
    float lo, hi;
};

NoOpacity no_opacity(const vbm_tf *tf)
{
    const float inf = std::numeric_limits<float>::infinity();
    const float absent = std::numeric_limits<float>::quiet_NaN();
    NoOpacity r{absent, absent};
    const int n = tf->n_knots;
    int k = 0;
    while (k < n && tf->rgba[k][3] <= 0.f) k++;
    if (k == n) return NoOpacity{inf, absent};               // no opacity anywhere
    if (k > 0 && tf->x[k - 1] >= 0.f) r.lo = tf->x[k - 1] * (1.f - 1e-5f);
    k = n - 1;
    while (k >= 0 && tf->rgba[k][3] <= 0.f) k--;
    if (k < n - 1 && tf->x[k + 1] <= 1.f) r.hi = std::max(tf->x[k + 1], 0.f) * (1.f + 1e-5f);
    return r;
}

// Occupancy words: bit b of word (bz, by, w) is block (32 w + b, by, bz).  One
// thread a column of x, over the 9 x 9 rows whose voxels are corners of the
// blocks' cells; a block then takes its 9 columns.  A voxel that is not
// comparable (NaN) counts as occupied, and so does one at or above kMarkMax, from
// which an interpolation can overflow: infinity times a weight of 0 is NaN and
// reads as the scalar 0.  (Below lo nothing need be excluded: a bound there
// means that 0 has no opacity either.)
//
// HIGH: the transfer function has an upper bound.  One that is opaque at its last
// knot has none, and its voxels take one comparison: the kernel is bound by
// their issue (image of 512^2 of 512^3 at a step of 1, 608 -> 592 us in all).
constexpr float kMarkMax = 1e38f;

template <bool HIGH>
__global__ void __launch_bounds__(kOccupancyThreads) k_occupancy(const float *__restrict__ F, int nx, int ny, int nz,
                                                                 NoOpacity none, uint32_t *__restrict__ words)
{
    __shared__ uint8_t low[kOccupancyCols + 1], high[kOccupancyCols + 1];
    const int x = blockIdx.x * kOccupancyCols + threadIdx.x;
    const int y0 = blockIdx.y * kCell, z0 = blockIdx.z * kCell;
    if (threadIdx.x <= kOccupancyCols) {
        bool lo = true, hi = HIGH;
        if (x < nx) {
            for (int z = z0; z <= min(z0 + kCell, nz - 1); z++) {
                const float *row = F + ((int64_t)z * ny + y0) * nx + x;
                float v[kCell + 1];
#pragma unroll
                for (int k = 0; k <= kCell; k++) v[k] = row[(int64_t)min(k, ny - 1 - y0) * nx];
#pragma unroll
                for (int k = 0; k <= kCell; k++) {
                    lo &= v[k] <= none.lo;
                    if (HIGH) hi &= v[k] >= none.hi && v[k] < kMarkMax;
                }
            }
        }
        low[threadIdx.x] = lo;
        high[threadIdx.x] = hi;
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    bool lo = true, hi = true;
#pragma unroll
    for (int k = 0; k <= kCell; k++) {
        lo &= low[threadIdx.x * kCell + k] != 0;
        hi &= high[threadIdx.x * kCell + k] != 0;
    }
    const uint32_t word = __ballot_sync(0xffffffffu, !lo && !hi);
    if (threadIdx.x == 0) words[((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = word;
}

// Lower cell corner and fraction of a clamped coordinate q (n voxels, last = n -
// 1).  Up to 2^23 voxels adding 2^23 rounding down leaves floor(q) in the low
// mantissa bits, without conversions (top: 2^23 + the last lower corner); the
// GENERAL march converts.
constexpr int kFloorMax = 1 << 23;
constexpr float kFloorMagic = (float)kFloorMax;
constexpr int kFloorBits = 0x4B000000;

template <bool GENERAL>
__device__ __forceinline__ int cell_of(float q, int n, float last, float top, float &frac)
{
    q = fminf(fmaxf(q, 0.f), last);
    if constexpr (GENERAL) {
        const int i = min((int)floorf(q), max(n - 2, 0));
        frac = q - (float)i;
        return i;
    }
    const float f = fminf(__fadd_rd(q, kFloorMagic), top);
    frac = q - (f - kFloorMagic);
    return __float_as_int(f) - kFloorBits;
}

// The march's roundings are spelled out, so that a ray's samples are the same
// bits whether or not it passes over empty blocks.  Near-parallel rays turn a
// last-bit change of their direction into 1e-4 of a pixel.
__device__ __forceinline__ float dot3(float a, float b, float c, float d, float e, float f)
{
    return __fmaf_rn(e, f, __fmaf_rn(a, b, __fmul_rn(c, d)));
}

__device__ __forceinline__ float mix(float a, float wa, float b, float wb)
{
    return __fmaf_rn(a, wa, __fmul_rn(b, wb));
}

// Transfer function and opacity correction as a ray evaluates them, in shared
// memory.  Interval k of the transfer function: x_k and 1 / (x_{k+1} - x_k),
// the colour at x_k and its change to the next knot.  corr: the Taylor
// polynomial of 1 - (1 - a)^step in (a - i / kCorr) kCorr about a = i / kCorr,
// good to 1.5e-9 for steps up to kMaxCorrStep and alphas below kMaxCorr; the
// last segment of a ray (shorter than the step), larger alphas and larger
// steps evaluate the power itself.  The images are as far from 64-bit ones as
// with a division an interval and the power of every sample (8 x 512^2 of 128^3
// 1.4e-6, 8 x 1024^2 of 512^3 3.2e-6).
constexpr int kDvrThreads = 128;             // 16 x 8 pixels: a block waits for its slowest ray (of 256: 454 us and 6.72
                                             // ms on 8 x 512^2 and 8 x 1024^2, of 128: 433 and 6.49, of 64: 460 and 6.77)
constexpr int kCorr = 256;
constexpr int kCorrCells = 192;
constexpr float kMaxCorr = (float)kCorrCells / kCorr;
constexpr float kMaxCorrStep = 4.f;

struct MarchTable {
    float4 rgba[16], change[16];
    float2 seg[16];
    float4 corr[kCorrCells];
};

__device__ __forceinline__ void march_stage(const TFDev &tf, float step, MarchTable &tab)
{
    int i = threadIdx.x;
    if (i < 16) {
        const int j = min(i + 1, 15);
        tab.rgba[i] = make_float4(tf.rgba[i][0], tf.rgba[i][1], tf.rgba[i][2], tf.rgba[i][3]);
        tab.change[i] = make_float4(tf.rgba[j][0] - tf.rgba[i][0], tf.rgba[j][1] - tf.rgba[i][1],
                                    tf.rgba[j][2] - tf.rgba[i][2], tf.rgba[j][3] - tf.rgba[i][3]);
        tab.seg[i] = make_float2(tf.x[i], 1.f / (tf.x[j] - tf.x[i]));
    }
    for (; i < kCorrCells; i += kDvrThreads) {
        const float a = (float)i / kCorr, log_rest = log1pf(-a), h = 1.f / kCorr, ratio = h / (1.f - a);
        const float c1 = step * expf((step - 1.f) * log_rest) * h;
        const float c2 = 0.5f * (1.f - step) * c1 * ratio;
        tab.corr[i] = make_float4(-expm1f(step * log_rest), c1, c2, (1.f / 3.f) * (2.f - step) * c2 * ratio);
    }
}

// Colour and opacity at the scalar f.
__device__ __forceinline__ float4 march_tf(const TFDev &tf, const MarchTable &tab, float f)
{
    f = fminf(fmaxf(f, 0.f), 1.f);
    if (f <= tf.x[0]) return tab.rgba[0];
    if (f >= tf.x[tf.n - 1]) return tab.rgba[tf.n - 1];
    int k = 0;
#pragma unroll
    for (int i = 0; i < 6; i++) k += tf.xs[i] <= f;
    if (tf.n > 8) {
#pragma unroll
        for (int i = 6; i < 14; i++) k += tf.xs[i] <= f;
    }
    const float2 seg = tab.seg[k];
    const float4 a = tab.rgba[k], c = tab.change[k];
    const float t = __fmul_rn(__fsub_rn(f, seg.x), seg.y);
    return make_float4(__fmaf_rn(t, c.x, a.x), __fmaf_rn(t, c.y, a.y), __fmaf_rn(t, c.z, a.z),
                       __fmaf_rn(t, c.w, a.w));
}

// SKIP: use the occupancy words.  GENERAL: any volume; otherwise every edge has 2
// to kFloorMax voxels and the volume less than 2^30 (32-bit byte offsets).
template <bool SKIP, bool GENERAL>
__global__ void __launch_bounds__(kDvrThreads) k_dvr(const float *__restrict__ F, int nx, int ny, int nz,
                                             const __grid_constant__ TFDev tf, NoOpacity none,
                                             const vbm_camera *__restrict__ cams, int W, int H, float step,
                                             const uint32_t *__restrict__ words, float *__restrict__ out)
{
    __shared__ MarchTable table;
    march_stage(tf, step, table);
    __syncthreads();
    const int v = blockIdx.z;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the image's blocks row by row along the grid's first axis, whose extent no
    // image reaches (the second holds 65535)
    const int block_cols = (W + 15) / 16, by = blockIdx.x / block_cols, bx = blockIdx.x - by * block_cols;
    const int px = bx * 16 + (warp & 1) * 8 + (lane & 7);
    const int py = by * (kDvrThreads / 16) + (warp >> 1) * 4 + (lane >> 3);
    const bool inside = px < W && py < H;                // every lane stays for the warp's votes
    const vbm_camera cam = cams[v];
    const float dcx = (px + 0.5f - cam.cx) / cam.fx, dcy = (py + 0.5f - cam.cy) / cam.fy;   // and 1 along z
    const float *R = cam.R;
    float d[3], o[3];
#pragma unroll
    for (int k = 0; k < 3; k++) d[k] = __fadd_rn(mix(R[k], dcx, R[3 + k], dcy), R[6 + k]);   // R^T dc
    const float inv_len = rsqrtf(dot3(d[0], d[0], d[1], d[1], d[2], d[2]));
#pragma unroll
    for (int k = 0; k < 3; k++) {
        d[k] *= inv_len;
        o[k] = -dot3(R[k], cam.t[0], R[3 + k], cam.t[1], R[6 + k], cam.t[2]);   // -R^T t
    }
    const int n[3] = {nx, ny, nz};
    const float box[3] = {(float)nx, (float)ny, (float)nz};
    float t0 = 0.f, t1 = 3.4e38f;
    bool miss = false;
    float inv_d[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        inv_d[k] = 0.f;
        if (d[k] != 0.f) {
            const float inv = 1.f / d[k];
            inv_d[k] = inv;
            float ta = (0.f - o[k]) * inv, tb = (box[k] - o[k]) * inv;
            t0 = fmaxf(t0, fminf(ta, tb));
            t1 = fminf(t1, fmaxf(ta, tb));
        } else if (o[k] < 0.f || o[k] > box[k]) {
            miss = true;
        }
    }
    float C0 = 0.f, C1 = 0.f, C2 = 0.f, T = 1.f;
    const bool hit = inside && !miss && t1 > t0;
    const int nseg = hit ? (int)ceilf((t1 - t0) / step) : 0;
    // Distance along the ray to a block's face: (8 c + face[k] - q[k]) inv_d[k] from
    // the position q in block c.  The face is taken `margin` too near, so that the
    // samples up to it lie in the block as their positions round.  A position is
    // the float32 of o + tm d - 1/2 with tm the float32 of t0 + (m + 1/2) step: two
    // samples' positions differ from the exact multiple of the step by at most 6
    // 2^-24 (t1 + n) together (three roundings up to t1 and two up to n voxels for
    // each), and 1e-5 covers the distance's own.  Towards the face they come in
    // order, so none falls back behind the block's other faces.
    // A ray that does not move along an axis leaves the block through neither
    // face: it looks at the one ahead of its q, infinitely far (a face at or behind
    // q sent such a ray's empty space through the occupancy words sample by
    // sample: 65536 x 16 x 16 at a step of 0.05, 200 -> 1.3 ms).
    float face[3] = {0.f, 0.f, 0.f};
    if (SKIP && nseg > 0) {
        const float margin = __fmaf_rn(0x1p-21f, t1 + fmaxf(fmaxf(box[0], box[1]), box[2]), 1e-5f);
#pragma unroll
        for (int k = 0; k < 3; k++) {
            if (d[k] != 0.f) {
                face[k] = d[k] > 0.f ? (float)kCell - margin : margin;
            } else {
                const bool up = o[k] - 0.5f <= fmaxf(box[k] - 2.f, 0.f);
                inv_d[k] = up ? 1e30f : -1e30f;
                face[k] = up ? (float)kCell : 0.f;
            }
        }
    }
    const float last[3] = {(float)(nx - 1), (float)(ny - 1), (float)(nz - 1)};
    // a cell's upper corner exists: the lower one is at most n - 2 (0 where n = 1)
    const float top[3] = {kFloorMagic + (float)max(nx - 2, 0), kFloorMagic + (float)max(ny - 2, 0),
                          kFloorMagic + (float)max(nz - 2, 0)};
    const float table_max = step <= kMaxCorrStep ? kMaxCorr : 0.f;   // alphas below it use the table
    const int64_t plane = (int64_t)nx * ny;
    const float *F10 = F + nx, *F01 = F + plane, *F11 = F01 + nx;
    const float inv_step = 1.f / step;
    const int word_cols = (nx + kOccupancyCols - 1) / kOccupancyCols, block_rows = (ny + kCell - 1) / kCell;
    // samples [m, m_end) lie in an occupied block; m = nseg: the ray is done
    int m = 0, m_end = SKIP ? 0 : nseg;
    // corners of the last sample's cell (fast path): at two samples a voxel the
    // next one lies in the same cell 40% of the time, and its lanes need no
    // loads (8 x 1024^2 of a 512^3 volume 7.15 -> 6.72 ms: the L1 wavefronts of
    // the corner loads bound it)
    uint32_t cell = 0xffffffffu;
    float2 k00 = make_float2(0.f, 0.f), k10 = k00, k01 = k00, k11 = k00;
    for (;;) {
        // 1. every ray that has left its block passes to its next occupied one
        if constexpr (SKIP) {
            while (__any_sync(0xffffffffu, m < nseg && m >= m_end)) {
                if (m >= nseg || m < m_end) continue;
                const float a0 = __fmaf_rn((float)m, step, t0), tm = __fmaf_rn(0.5f, fminf(step, t1 - a0), a0);
                float q[3], f;
                int c[3];
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    q[k] = __fadd_rn(__fmaf_rn(tm, d[k], o[k]), -0.5f);
                    c[k] = cell_of<GENERAL>(q[k], n[k], last[k], top[k], f) >> kCellShift;
                }
                // samples from m on that lie in this block for certain
                float leave = 1e6f;
#pragma unroll
                for (int k = 0; k < 3; k++)
                    leave = fminf(leave, (__fmaf_rn((float)kCell, (float)c[k], face[k]) - q[k]) * inv_d[k]);
                m_end = m + min(nseg - m, 1 + max(0, (int)fminf(leave * inv_step, 1e6f)));
                const uint32_t word = words[((int64_t)c[2] * block_rows + c[1]) * word_cols + (c[0] >> 5)];
                if (!((word >> (c[0] & 31)) & 1u)) m = m_end;
            }
        }
        // 2. one sample a round for every ray inside its block, until fewer
        // than three quarters of the unfinished ones still are
        const int enough = SKIP ? __popc(__ballot_sync(0xffffffffu, m < nseg)) * 3 / 4 : 0;
        int going;
        do {
            if (m < min(m_end, nseg)) {
                const float a0 = __fmaf_rn((float)m, step, t0);
                const float seg = fminf(step, t1 - a0);
                m++;
                if (seg > 0.f) {
                    const float tm = __fmaf_rn(0.5f, seg, a0);
                    float fx, fy, fz;
                    const int x = cell_of<GENERAL>(__fadd_rn(__fmaf_rn(tm, d[0], o[0]), -0.5f), n[0], last[0], top[0], fx);
                    const int y = cell_of<GENERAL>(__fadd_rn(__fmaf_rn(tm, d[1], o[1]), -0.5f), n[1], last[1], top[1], fy);
                    const int z = cell_of<GENERAL>(__fadd_rn(__fmaf_rn(tm, d[2], o[2]), -0.5f), n[2], last[2], top[2], fz);
                    const float gx = 1.f - fx, gy = 1.f - fy;
                    float c00, c10, c01, c11;
                    if constexpr (GENERAL) {
                        const float *p = F + (((int64_t)z * ny + y) * nx + x), *r = p + (nz > 1 ? plane : 0);
                        const int dx = nx > 1, dy = ny > 1 ? nx : 0;
                        c00 = mix(p[0], gx, p[dx], fx), c10 = mix(p[dy], gx, p[dy + dx], fx);
                        c01 = mix(r[0], gx, r[dx], fx), c11 = mix(r[dy], gx, r[dy + dx], fx);
                    } else {
                        const uint32_t at = ((uint32_t)(z * ny + y) * nx + x) * 4u;
                        if (at != cell) {
                            cell = at;
                            auto row = [&](const float *f) {
                                const float *p = reinterpret_cast<const float *>(reinterpret_cast<const char *>(f) + at);
                                return make_float2(p[0], p[1]);
                            };
                            k00 = row(F), k10 = row(F10), k01 = row(F01), k11 = row(F11);
                        }
                        c00 = mix(k00.x, gx, k00.y, fx), c10 = mix(k10.x, gx, k10.y, fx);
                        c01 = mix(k01.x, gx, k01.y, fx), c11 = mix(k11.x, gx, k11.y, fx);
                    }
                    const float val = mix(mix(c00, gy, c10, fy), 1.f - fz, mix(c01, gy, c11, fy), fz);
                    if (!(val <= none.lo || val >= none.hi)) {       // otherwise no opacity
                        const float4 rgba = march_tf(tf, table, val);
                        if (rgba.w > 0.f) {
                            float ac = 1.f;
                            if (seg == step && rgba.w < table_max) {
                                const float u = rgba.w * kCorr, i = floorf(u), e = u - i;
                                const float4 c = table.corr[(int)i];
                                ac = __fmaf_rn(e, __fmaf_rn(e, __fmaf_rn(e, c.w, c.z), c.y), c.x);
                            } else if (rgba.w < 1.f) {
                                ac = -expm1f(seg * log1pf(-rgba.w));
                            }
                            const float wgt = T * ac;
                            C0 = __fmaf_rn(wgt, rgba.x, C0);
                            C1 = __fmaf_rn(wgt, rgba.y, C1);
                            C2 = __fmaf_rn(wgt, rgba.z, C2);
                            T *= 1.f - ac;
                            if (T < 1e-6f) m = nseg;
                        }
                    }
                } else {
                    m = nseg;
                }
            }
            going = __popc(__ballot_sync(0xffffffffu, m < min(m_end, nseg)));
        } while (going > enough);
        if (going == 0 && !__any_sync(0xffffffffu, m < nseg)) break;
    }
    if (!inside) return;
    const int64_t HW = (int64_t)H * W, pix = (int64_t)py * W + px;
    out[((int64_t)v * 4 + 0) * HW + pix] = C0;
    out[((int64_t)v * 4 + 1) * HW + pix] = C1;
    out[((int64_t)v * 4 + 2) * HW + pix] = C2;
    out[((int64_t)v * 4 + 3) * HW + pix] = 1.f - T;
}

dim3 occupancy_grid(const int dims[3])
{
    return dim3((dims[0] + kOccupancyCols - 1) / kOccupancyCols, (dims[1] + kCell - 1) / kCell,
                (dims[2] + kCell - 1) / kCell);
}

}  // namespace

size_t dvr_workspace_bytes(const int dims[3])
{
    const dim3 g = occupancy_grid(dims);
    return (size_t)g.x * g.y * g.z * sizeof(uint32_t);
}

// ws: dvr_workspace_bytes(dims) of scratch, or NULL for a march without the
// occupancy marks.
vbm_status render_dvr(const float *F, const int dims[3], const vbm_tf *tf, const vbm_camera *cams, int n_views,
                      int W, int H, float step, float *out, void *ws, cudaStream_t st)
{
    const TFDev t = to_dev(tf);
    const NoOpacity none = no_opacity(tf);
    const dim3 marks = occupancy_grid(dims);
    uint32_t *words = (uint32_t *)ws;
    if (marks.y > 65535 || marks.z > 65535) words = nullptr;     // beyond a grid's extent
    const int64_t blocks = (int64_t)((W + 15) / 16) * ((H + kDvrThreads / 16 - 1) / (kDvrThreads / 16));
    VBM_ARG(blocks <= INT_MAX, "image too large");
    dim3 grid((unsigned)blocks, 1, n_views);
    const bool general = std::min({dims[0], dims[1], dims[2]}) < 2 ||
                         std::max({dims[0], dims[1], dims[2]}) > kFloorMax ||
                         (int64_t)dims[0] * dims[1] * dims[2] >= (int64_t)1 << 30;
    if (words) {
        auto occupancy = none.hi == none.hi ? k_occupancy<true> : k_occupancy<false>;
        occupancy<<<marks, kOccupancyThreads, 0, st>>>(F, dims[0], dims[1], dims[2], none, words);
        VBM_LAUNCH("occupancy");
        note_launches(1);
    }
    auto kernel = words ? (general ? k_dvr<true, true> : k_dvr<true, false>)
                        : (general ? k_dvr<false, true> : k_dvr<false, false>);
    kernel<<<grid, kDvrThreads, 0, st>>>(F, dims[0], dims[1], dims[2], t, none, cams, W, H, step, words, out);
    VBM_LAUNCH("render_dvr");
    note_launches(1);
    return VBM_OK;
}

}  // namespace vbm
