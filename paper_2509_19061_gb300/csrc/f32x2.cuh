// f32x2.cuh -- packed FP32 pairs (internal): two FP32 values in one 64-bit
// register pair, operated on by one instruction of sm_100-class GPUs, and the
// column shuffles of the kernels whose lanes own two adjacent columns.
#pragma once

#include <cuda_runtime.h>

namespace stokes {

struct f2 {
    unsigned long long u;
};
__device__ __forceinline__ f2 pk(float lo, float hi)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.u) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float f2lo(f2 a)
{
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.u));
    return x;
}
__device__ __forceinline__ float f2hi(f2 a)
{
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.u));
    return y;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b)
{
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b)
{
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.u) : "l"(a.u), "l"(b.u), "l"(c.u));
    return r;
}
// a * b rounded once and never fused into a following addition: the code
// generator contracts mul.rn.f32x2 followed by add/sub.rn.f32x2 into one
// fused multiply-add despite the rounding modifier (measured: a packed
// product minus a nearly equal value differs from the scalar rounded
// sequence in almost every case), so the product is formed as
// fma(a, b, +0), which rounds a * b once and is not contracted.  Its only
// difference from a plain product is the sign of an exact zero (+0 for -0).
__device__ __forceinline__ f2 mul2r(f2 a, f2 b)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.u) : "l"(a.u), "l"(b.u), "l"(0ull));
    return r;
}
// (x(c0 - 1), x(c0)) and (x(c1), x(c1 + 1)) of a pair (x(c0), x(c1))
__device__ __forceinline__ f2 west_pair(f2 a) { return pk(__shfl_up_sync(0xffffffffu, f2hi(a), 1), f2lo(a)); }
__device__ __forceinline__ f2 east_pair(f2 a) { return pk(f2hi(a), __shfl_down_sync(0xffffffffu, f2lo(a), 1)); }

} // namespace stokes
