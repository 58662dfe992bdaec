// packed.cuh -- packed FP32x2 helpers: a complex64 amplitude as one 64-bit register.
#pragma once
#include <cuda_runtime.h>

namespace qsim {

typedef unsigned long long u64;

__device__ __forceinline__ u64 pk(float x, float y) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}

// packed FP32x2 FMA on register pairs
__device__ __forceinline__ u64 fma2p(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ float2 unpk(u64 w) {
    float2 v;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(w));
    return v;
}

// v * i^k
__device__ __forceinline__ float2 mul_ipow(float2 v, int k) {
    float2 r = (k & 1) ? make_float2(-v.y, v.x) : v;
    if (k & 2) { r.x = -r.x; r.y = -r.y; }
    return r;
}

}  // namespace qsim
