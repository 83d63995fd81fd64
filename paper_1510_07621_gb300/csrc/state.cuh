// Particle-state helpers of the load and key kernels, without FP64 arithmetic in the common case: an
// FP64 instruction takes about 17 cycles per warp on a GB300 SM, so that three compares per coordinate
// kept these kernels on the FP64 pipe (80 to 86 % busy) where memory is their floor.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace {

// x = fmod(x, L); x < 0 -> x += L; x >= L -> x -= L.  (fmod(x, L) == x for -L < x < L)
// Not inlined: the compiler would otherwise run the compares for every particle.
__device__ __noinline__ double wrap_box_outside(double x, double L)
{
    if (!(x > -L && x < L)) x = fmod(x, L);
    if (x < 0.0) x = __dadd_rn(x, L);
    if (x >= L) x = __dadd_rn(x, -L);
    return x;
}

// x inside [0, L) (the common case after a drift) as one integer compare of the bit patterns (IEEE
// order of non-negative doubles); -0.0, NaN and negative x have larger patterns and take the full
// sequence, which leaves -0.0 unchanged.
__device__ __forceinline__ double wrap_box(double x, double L)
{
    if ((unsigned long long)__double_as_longlong(x) < (unsigned long long)__double_as_longlong(L)) return x;
    return wrap_box_outside(x, L);
}

// isfinite by the exponent bits
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7FF00000) != 0x7FF00000; }

}  // namespace
