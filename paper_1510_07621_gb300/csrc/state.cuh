// Particle-state helpers of the load, key and mesh kernels, without FP64 arithmetic where it can be had: an
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

// i = floor(u) and f = u - i, both exact, for 0 <= u < 4096 (mesh coordinates; any other value: i = 0).
// One FP64 instruction: the fraction's bits behind a 1 are 1 + f.  floor, conversion and difference take
// three (128^3 FP64: gather 0.196 -> 0.174 ms, deposit 0.144 -> 0.122).
__device__ __forceinline__ void split_floor(double u, int &i, double &f)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(u);
    const int e = (int)(b >> 52) - 1023;  // u in [2^e, 2^(e + 1))
    const unsigned long long frac = (b << (e & 15)) & 0xFFFFFFFFFFFFFull;
    const double g = __longlong_as_double((long long)(frac | 0x3FF0000000000000ull)) - 1.0;
    const unsigned int top = (unsigned int)(b >> 32) & 0xFFFFFu;  // the leading 20 bits after the 1
    const bool whole = e >= 0 && e < 12;
    i = whole ? (int)((top | 0x100000u) >> (20 - (e & 15))) : 0;
    f = whole ? g : u;
}

}  // namespace
