// da_fixed.cuh -- conversions between fp32 and the fixed-point grid 2^-S of
// the exact field recompute, in integer arithmetic.
//
// The recompute's definition is  v = round(w 2^S)  (to nearest, ties to even)
// for every coefficient and  g = fl32(sum) 2^-S  for every field.  Written with
// the 64-bit conversions of the instruction set (__float2ll_rn, __ll2float_rn)
// those run on the fp64 pipe, which is a small fraction of the fp32 rate on
// this GPU; the versions below use the integer and fp32 pipes only and return
// the same bits for every argument the recompute produces.
#pragma once
#include <cstdint>

namespace da {

// round(w 2^S) for finite w with |w 2^S| < 2^63; equal to
// __float2ll_rn(ldexpf(w, S)) (values whose scaled magnitude is below 1/2,
// including those that ldexpf would round to subnormals, give 0 both ways).
__device__ __forceinline__ long long fixed_of_f32(float w, int S)
{
    const uint32_t b = __float_as_uint(w);
    const uint32_t E = (b >> 23) & 0xFFu;
    const uint32_t m = E ? ((b & 0x7FFFFFu) | 0x800000u) : (b & 0x7FFFFFu);
    const int sh = (E ? (int)E : 1) - 150 + S;   // |w| 2^S = m 2^sh
    unsigned long long mag;
    if (sh >= 0) {
        mag = (unsigned long long)m << sh;
    } else if (sh <= -25) {
        mag = 0;                                 // m 2^sh < 1/2
    } else {
        const int rs = -sh;
        const uint32_t q = m >> rs;
        const uint32_t rem = m & ((1u << rs) - 1u);
        const uint32_t half = 1u << (rs - 1);
        mag = q + ((rem > half || (rem == half && (q & 1u))) ? 1u : 0u);
    }
    return (b >> 31) ? -(long long)mag : (long long)mag;
}

// fl32(v) 2^-S: v rounded to fp32 (to nearest, ties to even), then scaled;
// equal to ldexpf(__ll2float_rn(v), -S).  |v| is shifted so that its leading bit is
// bit 31 of a 32-bit word whose lowest bit also stands for all bits below it: the
// word's conversion then rounds as the 64-bit value would, and the scale is a
// multiplication by a power of two.  Scales outside the normal range are left to
// ldexpf.
__device__ __forceinline__ float scaled_f32_of(long long v, int S)
{
    const unsigned long long u = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int z = __clzll((long long)u);         // 64 for v = 0
    const unsigned long long n = u << (z & 63);
    const uint32_t top = (uint32_t)(n >> 32) | ((uint32_t)n != 0u ? 1u : 0u);
    const float f = __uint_as_float(__float_as_uint(__uint2float_rn(top)) | (v < 0 ? 0x80000000u : 0u));
    const int x = 32 - z - S;                     // |v| 2^-S = top 2^x
    // the product stays normal: top is 0 or at least 2^31, at most 2^32
    if (x >= -126 && x <= 95) return v == 0 ? 0.f : __fmul_rn(f, __uint_as_float((uint32_t)(x + 127) << 23));
    return v == 0 ? 0.f : ldexpf(f, x);
}

// The energy (hi 2^64 + lo) / 2^(S + 1) of a 128-bit sum: integer couplings (S = 0) as
// int64 (exact), fp32 ones rounded once to fp64, as its bits.
template <bool INT8>
__device__ __forceinline__ long long energy_of_sum(unsigned long long lo, long long hi, int S)
{
    if constexpr (INT8) {
        return (long long)lo / 2;   // |2E| < 2^63
    } else {
        // value = hi 2^64 + lo; top = value >> 32 (exact in fp64, |value| < 2^76)
        const long long top = (long long)((unsigned long long)hi << 32 | (lo >> 32));
        const double bottom = (double)(uint32_t)(lo & 0xFFFFFFFFull);
        const double v = __fma_rn((double)top, 4294967296.0, bottom);
        return __double_as_longlong(ldexp(v, -(S + 1)));
    }
}

// The integer value of an fp32 that holds an integer in [-2^22, 2^22)
// (the tensor cores' digit sums): adding 1.5 2^23 puts it in the mantissa.
__device__ __forceinline__ int small_int_of(float f)
{
    return __float_as_int(__fadd_rn(f, 12582912.0f)) - 0x4B400000;
}

}  // namespace da
