// FP32 hardware approximations without the denormal handling of the CUDA
// functions (about 2^-22 relative for the reciprocal square root; sine and cosine
// to about 2^-21 absolute on [-pi, pi], where the callers reduce the phase to).
#pragma once

#include <cuda_runtime.h>

namespace ibem {

__device__ __forceinline__ float approx_rsqrt(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float approx_sin(float x) {
    float y;
    asm("sin.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float approx_cos(float x) {
    float y;
    asm("cos.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// x - 2 pi round(x / (2 pi)); adding 1.5 2^23 rounds (on the FMA pipe, unlike rintf)
__device__ __forceinline__ float reduce_phase(float x) {
    const float n = fmaf(x, 0.15915494309189535f, 12582912.0f) - 12582912.0f;
    return fmaf(-6.283185307179586f, n, x);
}

}  // namespace ibem
