// fixed_dot.cuh -- FP64 dot products as exact integer sums.
//
// sum_k m_k v_k with |m| < 2^em, |v| < 2^ev: both become integers of `bits` bits (rounded once,
// 2^-bits of their bounds), each two balanced digits, the lower one of `lob` bits (28 unless
// said otherwise), and three 32 x 32 + 64 -> 64 multiply-adds per entry sum
// hi hi' 2^(2 lob) + (hi lo' + lo hi') 2^lob exactly (lo lo' lies below the last bit kept).  The
// sum is value() * 2^(em + ev - 2 bits + 2 lob).  One multiply-add takes a warp 1 clock of its
// SM's integer pipes; an FP64 multiply-add takes 19.
#pragma once

#include "common.cuh"

namespace uoi {

// rint(x 2^(bits - e)) for |x| < 2^e as two digits.
__device__ __forceinline__ int2 fx_digits(double x, int e, int bits, int lob = 28)
{
    const long long b = __double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7FF);
    long long q = b & 0xFFFFFFFFFFFFFll;
    if (ex) q |= 1ll << 52;
    const int sh = max(ex, 1) - 1075 + bits - e;          // at most bits - 53
    if (sh >= 0) q <<= sh;
    else if (sh < -54) q = 0;
    else q = (q + (1ll << (-sh - 1))) >> -sh;
    if (b < 0) q = -q;
    const long long hi = (q + (1ll << (lob - 1))) >> lob;
    return make_int2((int)hi, (int)(q - (hi << lob)));
}

// e with |x| < 2^e for values whose high word (without sign) is at most h.
__device__ __forceinline__ int fx_exponent(uint32_t h) { return max((int)(h >> 20), 1) - 1022; }

// High word of |x|, 1 for a subnormal that lies in the low word alone.
__device__ __forceinline__ uint32_t fx_high(double x)
{
    const uint32_t h = (uint32_t)__double2hiint(x) & 0x7FFFFFFFu;
    return h == 0 && __double2loint(x) != 0 ? 1u : h;
}

// Sum of products; value(): the sum in units of 2^(2 lob), rounded.
struct FxSum {
    using Out = long long;
    long long hh = 0, mid = 0;
    __device__ __forceinline__ void add(int2 m, int2 v)
    {
        hh += (long long)m.x * v.x;
        mid += (long long)m.x * v.y;
        mid += (long long)m.y * v.x;
    }
    __device__ __forceinline__ long long value(int lob = 28) const { return hh + ((mid + (1ll << (lob - 1))) >> lob); }
};

// All four products: the sum is hh 2^(2 lob) + low(lob), the first exact, the second rounded at
// 2^-53 of itself.
struct FxFull {
    long long hh = 0, mid = 0, ll = 0;
    __device__ __forceinline__ void add(int2 m, int2 v)
    {
        hh += (long long)m.x * v.x;
        mid += (long long)m.x * v.y;
        mid += (long long)m.y * v.x;
        ll += (long long)m.y * v.y;
    }
    __device__ __forceinline__ double low(int lob) const { return fma((double)mid, (double)(1ll << lob), (double)ll); }
};

// 2^e for any e that FP64 can hold (0 or Inf past its range).
__device__ __forceinline__ double fx_pow2(int e)
{
    return e > -1023 && e < 1024 ? __longlong_as_double((long long)(e + 1023) << 52) : scalbn(1.0, e);
}

// b - 2^e (hh 2^(2 lob) + low): the digits of hh go in one after the other, so that nothing but
// the result is rounded where it cancels against b.
__device__ __forceinline__ double fx_residual(double b, long long hh, double low, int e, int lob)
{
    b = fma(-fx_pow2(e + 2 * lob + 32), (double)(int)(hh >> 32), b);
    b = fma(-fx_pow2(e + 2 * lob), (double)(uint32_t)hh, b);
    return fma(-fx_pow2(e), low, b);
}

}  // namespace uoi
