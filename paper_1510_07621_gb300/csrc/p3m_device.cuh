// Device helpers of the FP32 pair kernels (short-range force and its reverse-mode derivative): the
// MUFU functions and packed two-lane FP32 arithmetic (f32x2) of sm_100-class GPUs.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace {

__device__ __forceinline__ float rsqrt_approx(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 2^x (MUFU)
__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Packed two-lane FP32 values (f32x2) through the compiler's own float2 builtins, so that
// register pairs and scheduling are the compiler's to choose.
typedef float2 f2;

__device__ __forceinline__ f2 f2_pack(float lo, float hi) { return make_float2(lo, hi); }
__device__ __forceinline__ void f2_unpack(f2 v, float &lo, float &hi)
{
    lo = v.x;
    hi = v.y;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 f2_neg(f2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }

}  // namespace
