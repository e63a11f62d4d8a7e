// fr_fp64.cuh -- FP64 helpers that spare this GPU's FP64 pipe.
//
// Measured on the GB300: an FP64 add, multiply, FMA or integer conversion
// occupies its SM sub-partition for 64 cycles (76 with every sub-partition
// busy), not pipelined and whatever the number of active lanes, and a double
// division is eight of them (580 cycles).  So the episode statistics and the
// indicator chains are paced by the number of FP64 warp instructions, and
// what the integer pipe can do exactly is done there.  Every helper returns
// the same bits as the plain FP64 operation that it stands for.
#pragma once

#include <stdint.h>

namespace fr {

// (double)x of an integer 0 <= x < 2^53 (exact, so no rounding is involved),
// assembled on the integer pipe: exponent from the leading bit, the bits
// below it as the fraction.
__device__ __forceinline__ double u53_to_double(uint64_t x)
{
    const int lead = 63 - __clzll((long long)x);           // -1 for 0
    const uint64_t frac = (x << ((52 - lead) & 63)) & 0xfffffffffffffull;
    const uint64_t bits = ((uint64_t)(uint32_t)(1023 + lead) << 52) | frac;
    return x == 0 ? 0.0 : __longlong_as_double((long long)bits);
}

// The plain operations, out of line: what the fast forms fall back to is rare,
// and inline the compiler would run its conversions on every call.
static __device__ __noinline__ double fp64_of_int(int64_t x) { return (double)x; }
static __device__ __noinline__ double fp64_div_int(double z, uint32_t n) { return __ddiv_rn(z, (double)n); }
static __device__ __noinline__ double fp64_int_ratio(int64_t a, int64_t b) { return __ddiv_rn((double)a, (double)b); }

// (double)x for any int64: the conversion instruction outside [0, 2^53).
__device__ __forceinline__ double i64_to_double(int64_t x)
{
    return ((uint64_t)x >> 53) == 0 ? u53_to_double((uint64_t)x) : fp64_of_int(x);
}

// An unevaluated sum hi + lo close to 1 / n.
struct Recip {
    double hi, lo;
};

// z / n, correctly rounded, by two operations in place of a division, for an
// integer 1 <= n < 2^31 and hi + lo = 1 / n to a relative error e <= 2^-88
// (the multiplication by an unevaluated sum of Brisebarre and Muller,
// "Correctly rounded multiplication by arbitrary precision constants", 2008).
// The value the FMA rounds is z / n (1 + d), |d| <= e + 2^-98.  z / n is never a
// midpoint between doubles (that would make z = n (2k + 1) 2^f with a 54-bit
// odd 2k + 1, more bits than z has) and its distance from one is at least
// 2^-54 / n > 2^-85 relative, so the rounding is that of z / n.  z outside
// [2^-900, 2^900) (zero apart, where both terms are exact) takes the
// division: the argument needs every term normal.
__device__ __forceinline__ bool div_recip_ok(double z)
{
    const uint32_t h = (uint32_t)__double2hiint(z), e = h & 0x7fffffffu;
    return e - ((1023u - 900u) << 20) < (1800u << 20) || (h | (uint32_t)__double2loint(z)) == 0u;
}

// The two operations alone, for a caller that knows z to be in range.  A
// chain checks that from what enters a group of steps and not on each z: an
// integer instruction between two dependent FP64 ones costs the chain a
// whole FP64 slot (measured: 383 cycles per Wilder step with the check on z,
// 258 without).
__device__ __forceinline__ double div_recip_fast(double z, Recip r)
{
    return __fma_rn(z, r.hi, __dmul_rn(z, r.lo));
}

__device__ __forceinline__ double div_recip(double z, Recip r, uint32_t n)
{
    const double q = div_recip_fast(z, r);
    return div_recip_ok(z) ? q : fp64_div_int(z, n);
}

// 1 / n as hi + lo for an integer 1 <= n < 2^31 given exactly as nd: a
// single-precision reciprocal (22 bits after both roundings), one Newton step
// (hi: 44 bits) and the residual 1 - n hi, which is exact (below 2^-44, its
// lowest bit 2^-84 or higher), times hi: relative error below 2^-88.
__device__ __forceinline__ Recip recip_of(uint32_t n, double nd)
{
    float r0;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(__uint2float_rn(n)));
    // the float's bits as a double's: exponent re-biased, fraction shifted
    const uint32_t b = __float_as_uint(r0);
    const double r = __hiloint2double((int)((b >> 3) + ((1023u - 127u) << 20)), (int)(b << 29));
    Recip out;
    out.hi = __fma_rn(r, __fma_rn(-nd, r, 1.0), r);
    out.lo = __dmul_rn(__fma_rn(-nd, out.hi, 1.0), out.hi);
    return out;
}

// v1 / v0, correctly rounded: six operations when 1 <= v0 < 2^31 and
// 0 <= v1 < 2^53, else the division.
__device__ __forceinline__ bool i64_ratio_fast(int64_t v1, int64_t v0)
{
    return v0 >= 1 && v0 < ((int64_t)1 << 31) && ((uint64_t)v1 >> 53) == 0;
}

__device__ __forceinline__ double i64_ratio(int64_t v1, int64_t v0)
{
    if (i64_ratio_fast(v1, v0)) {
        const double nd = u53_to_double((uint64_t)v0);
        return div_recip(u53_to_double((uint64_t)v1), recip_of((uint32_t)v0, nd), (uint32_t)v0);
    }
    return fp64_int_ratio(v1, v0);
}

// a / b < c / d for 0 <= a, c and 1 <= b, d, by 128-bit cross products.
__device__ __forceinline__ bool ratio_less(uint64_t a, uint64_t b, uint64_t c, uint64_t d)
{
    const uint64_t lh = __umul64hi(a, d), rh = __umul64hi(c, b);
    return lh < rh || (lh == rh && a * d < c * b);
}

}  // namespace fr
