// Transfer function on the device (Sec. 3): piecewise-linear RGBA of a scalar
// clamped to [0, 1], constant outside the knots.
#pragma once

#include "vbm_internal.h"

namespace vbm {

struct TFDev {
    int n;
    float x[16];
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
    return t;
}

#ifdef __CUDACC__
// The interpolation (1 - t) a + t b has its roundings spelled out, so every
// kernel that applies the transfer function gives the same bits.  `rgba` holds
// the knot colours in shared memory (a lane's knot index differs from its
// neighbours', which constant memory would serialise); the knot positions are
// read from the argument, where every lane compares with the same one.
__device__ __forceinline__ float4 tf_apply(const TFDev &tf, const float4 *rgba, float f)
{
    f = fminf(fmaxf(f, 0.f), 1.f);
    if (f <= tf.x[0]) return rgba[0];
    if (f >= tf.x[tf.n - 1]) return rgba[tf.n - 1];
    int k = 0;
    float xa = tf.x[0], xb = tf.x[1];
    for (int i = 1; i < tf.n - 1; i++) {
        const bool above = tf.x[i] <= f;
        k = above ? i : k;
        xa = above ? tf.x[i] : xa;
        xb = above ? tf.x[i + 1] : xb;
    }
    const float t = __fdiv_rn(__fsub_rn(f, xa), __fsub_rn(xb, xa)), s = __fsub_rn(1.f, t);
    const float4 a = rgba[k], b = rgba[k + 1];
    return make_float4(__fmaf_rn(s, a.x, __fmul_rn(t, b.x)), __fmaf_rn(s, a.y, __fmul_rn(t, b.y)),
                       __fmaf_rn(s, a.z, __fmul_rn(t, b.z)), __fmaf_rn(s, a.w, __fmul_rn(t, b.w)));
}

// Copies the knot colours to shared memory; the caller's next barrier publishes them.
__device__ __forceinline__ void tf_stage(const TFDev &tf, float4 (&rgba)[16])
{
    if (threadIdx.x < 16) {
        const float *c = tf.rgba[threadIdx.x];
        rgba[threadIdx.x] = make_float4(c[0], c[1], c[2], c[3]);
    }
}
#endif

}  // namespace vbm
