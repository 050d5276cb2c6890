// sbh_f32x2.cuh -- pairs of FP32 values in one 64-bit register, for Blackwell's packed
// instructions (add / mul / fma .rn.f32x2): each half is rounded as the scalar instruction rounds
// it. Measured on this chip a packed FMA takes the FMA pipe for two scalar ones' time (2.15
// cycles per warp and scheduler against 1.12), but one issue slot instead of two, which is what a
// loop that also issues loads, reciprocal roots and selects runs out of.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sbh {

struct f2 {
    uint64_t v;
};
__device__ __forceinline__ f2 f2_make(float lo, float hi)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ f2 f2_dup(float x) { return f2_make(x, x); }
__device__ __forceinline__ float f2_lo(f2 a)
{
    return __uint_as_float((uint32_t)a.v);
}
__device__ __forceinline__ float f2_hi(f2 a)
{
    return __uint_as_float((uint32_t)(a.v >> 32));
}
__device__ __forceinline__ f2 operator+(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 operator*(f2 a, f2 b)
{
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

}  // namespace sbh
