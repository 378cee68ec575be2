// Two FP32 values in a register pair and the packed operations on them: one issue
// slot for both, each half rounded as the scalar operation rounds it.  The two
// components of a voxel or a ray are such a pair.
#pragma once

#include <cuda_runtime.h>

namespace deam {

typedef unsigned long long pair32;

__device__ __forceinline__ pair32 pack2(float x, float y) {
    pair32 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ pair32 dup2(float x) { return pack2(x, x); }
__device__ __forceinline__ float2 unpack2(pair32 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
// a b + c
__device__ __forceinline__ pair32 fma2(pair32 a, pair32 b, pair32 c) {
    pair32 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ pair32 add2(pair32 a, pair32 b) {
    pair32 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ pair32 sub2(pair32 a, pair32 b) {
    pair32 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

}  // namespace deam
