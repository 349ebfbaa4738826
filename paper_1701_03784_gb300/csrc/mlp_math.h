// Elementwise arithmetic and copies of the surrogate networks, shared by the FP32 kernels.
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

// ---- asynchronous copies global -> shared ----------------------------------------------
// 16 or 4 bytes, of which the first `bytes` are read and the rest become zeros
__device__ __forceinline__ void cp16(float *dst, const float *src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp4(float *dst, const float *src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

}  // namespace pic
