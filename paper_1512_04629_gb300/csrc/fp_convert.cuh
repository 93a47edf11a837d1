// fp_convert.cuh -- FP32 <-> FP64 conversions that leave the FP64 pipe alone.
#pragma once
#include <stdint.h>

namespace amg {

// Conversions between the cycle's FP32 and the outer loop's FP64 on the integer
// pipes, exact and to nearest even: a conversion instruction holds the FP64
// pipe for 16 clocks as an FMA does -- also when it is predicated off, so the
// rare cases below are calls, which the compiler cannot turn into predicates.
// Every element of an outer iteration is widened twice and rounded once; on
// the conversion instructions the batched r.z pass of 45 M elements took
// 260 us, twice its memory time.
static __device__ __noinline__ double widen_rare(float f) { return (double)f; }
static __device__ __noinline__ float narrow_rare(double x) { return (float)x; }

__device__ __forceinline__ double widen(float f) {
    const uint32_t u = __float_as_uint(f), m = u & 0x7fffffffu;
    if (m - 0x00800000u >= 0x7f000000u && m != 0u) return widen_rare(f);  // subnormal, infinite, NaN
    const uint32_t hi = (u & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u);
    return __hiloint2double((int)hi, (int)(u << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }

// FP32 has 29 fewer fraction bits and an exponent bias 896 lower; rounding up
// carries into the exponent and, from the largest, to infinity
__device__ __forceinline__ float narrow(double x) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x), m = u & 0x7fffffffffffffffull;
    const uint32_t e = (uint32_t)(m >> 52);
    if (e - 897u > 253u && m != 0ull) return narrow_rare(x);  // outside FP32's normal range
    const uint32_t r = (uint32_t)((m + 0x0fffffffull + ((m >> 29) & 1ull)) >> 29) - (896u << 23);
    return __uint_as_float((uint32_t)(u >> 32 & 0x80000000u) | (m ? r : 0u));
}

}  // namespace amg
