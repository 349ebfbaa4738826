// Elementwise arithmetic of the surrogate networks, shared by the FP32 kernels.
#pragma once

#include "pic_internal.h"

namespace pic {

constexpr float C_GELU = 0.7978845608028654f;   // sqrt(2/pi)

__device__ __forceinline__ float gelu(float z) {
    return 0.5f * z * (1.f + tanhf(C_GELU * (z + 0.044715f * z * z * z)));
}
__device__ __forceinline__ float gelu_grad(float z) {
    const float t = tanhf(C_GELU * (z + 0.044715f * z * z * z));
    return 0.5f * (1.f + t) + 0.5f * z * (1.f - t * t) * C_GELU * (1.f + 3.f * 0.044715f * z * z);
}

// Adam's step for one parameter
__device__ __forceinline__ void adam_step(const AdamArgs &a, float gi, float &p, float &m, float &v) {
    const float mi = a.b1 * m + (1.f - a.b1) * gi;
    const float vi = a.b2 * v + (1.f - a.b2) * gi * gi;
    m = mi;
    v = vi;
    p -= a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
}

}  // namespace pic
