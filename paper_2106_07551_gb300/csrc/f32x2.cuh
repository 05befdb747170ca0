// Packed fp32 pairs (fma.rn.f32x2 and the like) for the kernels that run fp32
// sums on the CUDA cores.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace malib {

// Packed fp32 pair helpers: fma.rn.f32x2 performs two independent IEEE fp32
// fused multiply-adds (round to nearest), so results equal scalar fmaf.
__device__ __forceinline__ unsigned long long f2_dup(float v) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ void f2_fma(unsigned long long& d, unsigned long long a,
                                       unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ float2 f2_split(unsigned long long v) {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
    return make_float2(lo, hi);
}
__device__ __forceinline__ unsigned long long f2_relu(unsigned long long v) {
    const float2 q = f2_split(v);
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(fmaxf(q.x, 0.f)), "f"(fmaxf(q.y, 0.f)));
    return r;
}

// max(v, 0) that keeps a NaN (fmaxf(NaN, 0) is 0).
__device__ __forceinline__ float relu_nan(float v) {
    float r;
    asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ unsigned long long f2_relu_nan(unsigned long long v) {
    const float2 q = f2_split(v);
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(relu_nan(q.x)), "f"(relu_nan(q.y)));
    return r;
}

__device__ __forceinline__ unsigned long long f2_pack(uint32_t lo, uint32_t hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
// Two fp32 additions, each rounded to nearest.
__device__ __forceinline__ unsigned long long f2_add(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

}  // namespace malib
