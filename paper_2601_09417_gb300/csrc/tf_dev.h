// Transfer function on the device (Sec. 3): piecewise-linear RGBA of a scalar
// clamped to [0, 1], constant outside the knots.
#pragma once

#include <limits>

#include "vbm_internal.h"

namespace vbm {

// x holds the knot positions; xs the inner ones (1 .. n - 2), padded with
// infinity, whose count at or below a value is its interval.
struct TFDev {
    int n;
    float x[16];
    float xs[14];
    float rgba[16][4];
};

inline TFDev to_dev(const vbm_tf *tf)
{
    TFDev t{};
    t.n = tf->n_knots;
    for (int i = 0; i < 16; i++) {
        t.x[i] = tf->x[i];
        for (int c = 0; c < 4; c++) t.rgba[i][c] = tf->rgba[i][c];
    }
    for (int i = 0; i < 14; i++) t.xs[i] = i < t.n - 2 ? t.x[i + 1] : std::numeric_limits<float>::infinity();
    return t;
}

#ifdef __CUDACC__
// Interval starts, lengths and knot colours in shared memory: a lane's
// interval differs from its neighbours', which constant memory would
// serialise.  The inner knots stay in the argument, where every lane compares
// with the same one.
struct TFTable {
    float4 rgba[16];
    float2 seg[16];      // x_k, x_{k+1} - x_k
};

// The caller's next barrier publishes the table.
__device__ __forceinline__ void tf_stage(const TFDev &tf, TFTable &tab)
{
    const int i = threadIdx.x;
    if (i < 16) {
        tab.rgba[i] = make_float4(tf.rgba[i][0], tf.rgba[i][1], tf.rgba[i][2], tf.rgba[i][3]);
        tab.seg[i] = make_float2(tf.x[i], i < 15 ? __fsub_rn(tf.x[i + 1], tf.x[i]) : 0.f);
    }
}

// The interpolation (1 - t) a + t b has its roundings spelled out, so every
// kernel that applies the transfer function gives the same bits.
__device__ __forceinline__ float4 tf_apply(const TFDev &tf, const TFTable &tab, float f)
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
    const float t = __fdiv_rn(__fsub_rn(f, seg.x), seg.y), s = __fsub_rn(1.f, t);
    const float4 a = tab.rgba[k], b = tab.rgba[k + 1];
    return make_float4(__fmaf_rn(s, a.x, __fmul_rn(t, b.x)), __fmaf_rn(s, a.y, __fmul_rn(t, b.y)),
                       __fmaf_rn(s, a.z, __fmul_rn(t, b.z)), __fmaf_rn(s, a.w, __fmul_rn(t, b.w)));
}
#endif

}  // namespace vbm
