// Packed FP32 arithmetic: two values in one register pair, one instruction for
// both (the results are those of the scalar operations).
#pragma once

#include <cuda_runtime.h>

namespace zm {

// two FP32 values in one register pair
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
constexpr f32x2 F32X2_MINUS1 = 0xbf800000bf800000ull;      // (-1, -1)
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, F32X2_MINUS1, a); }
__device__ __forceinline__ f32x2 neg2(f32x2 a) { return mul2(a, F32X2_MINUS1); }

}  // namespace zm
