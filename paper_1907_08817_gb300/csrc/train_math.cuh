// train_math.cuh -- the scalar steps that the training kernels on the CUDA cores share (Sec. "Training",
// Eq. (loss); Adam per Kingma & Ba), stated once so that each of them rounds them the same way. The kernels
// of width 64 (k_train_tc.cu) state the same steps themselves, with the contractions the compiler chooses.
#pragma once
#include "common.cuh"

namespace nns {

// loss term and upstream gradient of one sample with residual r
__device__ __forceinline__ void loss_term(float r, int loss, float delta, float inv_n, float &gy, float &lv) {
    if (loss == NNSORT_LOSS_HUBER) {
        const float ar = fabsf(r);
        lv = (ar <= delta) ? 0.5f * r * r : delta * ar - 0.5f * delta * delta;
        gy = (r > delta) ? delta : ((r < -delta) ? -delta : r);
    } else {
        lv = r * r;
        gy = 2.0f * r;
    }
    gy *= inv_n;
}

// one Adam step of one parameter, its contractions written out so that every kernel that includes this makes
// the same ones; c1, c2: bias corrections; mask: +1/-1 the sign to keep, 0 free
__device__ __forceinline__ float adam_step(float p, float g, float &ms, float &vs, float lr, float b1, float b2,
                                           float eps, float c1, float c2, float mask) {
    const float m = __fmaf_rn(1.0f - b1, g, __fmul_rn(b1, ms));
    const float v = __fmaf_rn(__fmul_rn(1.0f - b2, g), g, __fmul_rn(b2, vs));
    ms = m;
    vs = v;
    const float mh = m / c1, vh = v / c2;
    float np = p - lr * mh / (sqrtf(vh) + eps);
    if (mask * np < 0.0f) np = 0.0f;  // monotone projection
    return np;
}

}  // namespace nns
