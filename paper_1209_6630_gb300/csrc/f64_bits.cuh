// Conversions between FP64 and float pairs on the integer pipes.
//
// GB300's FP64 pipe takes a warp instruction every 16 cycles of an SM, and the
// conversions between FP64 and FP32 go through it: splitting a double into a
// float pair costs three of its instructions and an addition (64 cycles per 32
// values), which bounded kernels that only move data (k_gt_init 8.5 -> 3.8 ms, k_gt_final 7.3 -> 3.7;
// where the issue slots are the limit -- the epilogue of k_c15_mma, the slicing in k_vd_mma -- they
// were slower).  Here the same values
// are formed from the bits; operands outside the ranges named below take the
// floating-point expressions, so the results are equal everywhere.
#pragma once

#include "ff_math.cuh"

namespace qmc {

// ff::from_double(x): h = x rounded to FP32, l = x - h rounded to FP32.  Fast for 2^-60 <= |x| < 2^120.
__device__ __forceinline__ float2 split_f64(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned ex = (hi >> 20) & 0x7ffu;                 // biased by 1023
    if (ex - (1023u - 60u) >= 180u) return (hi << 1 | lo) ? ff::from_double(x) : make_float2(__uint_as_float(hi), 0.f);
    // 23 of the 52 fraction bits, then round to nearest even on the other 29
    unsigned f = ((ex - 896u) << 23) | __funnelshift_l(lo, hi & 0xfffffu, 3);
    const unsigned rem = lo & 0x1fffffffu;
    const unsigned up = (rem + (f & 1u) > 0x10000000u) ? 1u : 0u;
    f += up;                                                 // (a carry out of the fraction is the next binade)
    // x - h = (rem - up 2^29) 2^(ex - 1075), exactly; at most 2^28 in magnitude
    const int r = (int)rem - (int)(up << 29);
    const unsigned s = hi & 0x80000000u;
    const float l = __int2float_rn(s ? -r : r) * __uint_as_float((ex - 948u) << 23);   // 2^(ex - 1075)
    return make_float2(__uint_as_float(f | s), l);
}

// ff::val(x) = (double)h + (double)l.  Fast where 2^-75 <= |h| < 2^120, |l| <= 2^-24 of h's binade,
// and the sum stays in h's binade.
__device__ __forceinline__ double join_f64(float2 x)
{
    const unsigned hb = __float_as_uint(x.x);
    const unsigned eh = (hb >> 23) & 0xffu, fh = hb & 0x7fffffu;
    // l in units of the sum's last place, 2^(eh - 127 - 52); |L| <= 2^28
    const float L = x.y * __uint_as_float((306u - eh) << 23);   // 2^(179 - eh)
    const bool in = ((int)(hb ^ __float_as_uint(L))) < 0;       // l points towards zero
    if (eh - 52u >= 195u || !(fabsf(L) <= 268435456.f) || (in && fh == 0u)) return ff::val(x);
    const int d = __float2int_rn(fabsf(L));
    const long long m = ((long long)fh << 29) + (in ? -(long long)d : (long long)d);
    const unsigned long long b = ((unsigned long long)(hb & 0x80000000u) << 32) |
                                 (((unsigned long long)(eh + 896u) << 52) + (unsigned long long)m);
    return __longlong_as_double((long long)b);
}

// |x| as an integer that orders like it, 0 for NaN (as fmaxf passes a NaN over)
__device__ __forceinline__ unsigned long long abs_bits(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
    return b > 0x7ff0000000000000ull ? 0ull : b;
}

}  // namespace qmc
