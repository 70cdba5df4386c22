// f32x2.cuh -- two FP32 values in a 64-bit register, one instruction for both.
#pragma once

#include <cuda_runtime.h>

namespace qsim {

typedef unsigned long long pack2;

__device__ __forceinline__ pack2 pk(float x, float y)
{
    pack2 v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
    return v;
}
__device__ __forceinline__ float2 unpk(pack2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ pack2 fma2(pack2 a, pack2 b, pack2 c)
{
    pack2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ pack2 mul2(pack2 a, pack2 b)
{
    pack2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ pack2 dup(float x) { return pk(x, x); }

}  // namespace qsim
