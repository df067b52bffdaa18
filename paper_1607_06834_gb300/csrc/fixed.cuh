// 64-bit fixed-point arithmetic on the integer pipe (FMA build).
//
// GB300 issues FP64 at 2 lane-operations per SM and clock (1.7 measured), but
// 32-bit integer multiply-adds and shifts at 64 and additions at 128.  A
// product of two 62-bit fixed-point numbers takes three 32 x 32 -> 64
// multiply-adds, two shifts and the limb splits (about 8 integer
// instructions, 4 SM clocks a warp, against 16 to 19 for one FP64
// instruction), an addition two integer instructions.  Where the range of the
// operands is known, the arithmetic is also more accurate than binary64: the
// rounding unit is 2^-62 of the range instead of 2^-53 of the value.
//
// Fx<S> holds a number x with |x| < 2^S as the integer x 2^(62 - S).  Scales
// are compile-time constants; products add them.  Nothing wraps as long as
// every operand of a product stays below 2^62 in magnitude; callers test the
// values that the bounds of the inputs do not keep there (reciprocals by the
// lower end of in_window), and discard a result whose test failed.
#pragma once
#include <cuda_runtime.h>

namespace rok {
namespace fx {

template <int S>
struct Fx {
    long long v;
};

constexpr long long kOne62 = 1ll << 62;

// limbs of v = hi 2^31 + lo, 0 <= lo < 2^31
__device__ __forceinline__ int limb_hi(long long v) { return (int)(v >> 31); }
__device__ __forceinline__ int limb_lo(long long v) { return (int)v & 0x7fffffff; }
__device__ __forceinline__ long long wide(int a, int b) { return (long long)a * b; }

// (a b) >> 62, truncated towards minus infinity (error below 2 units: the
// low product's carry is left out)
__device__ __forceinline__ long long mul62(long long a, long long b)
{
    const int ah = limb_hi(a), al = limb_lo(a), bh = limb_hi(b), bl = limb_lo(b);
    const long long c = wide(ah, bl) + wide(al, bh);
    return wide(ah, bh) + (c >> 31);
}

// (a b) >> (62 - K): K more bits of the product kept, for a result known to be
// below 2^-K of the product of the scales
template <int K>
__device__ __forceinline__ long long mul62k(long long a, long long b)
{
    const int ah = limb_hi(a), al = limb_lo(a), bh = limb_hi(b), bl = limb_lo(b);
    const long long c = wide(ah, bl) + wide(al, bh) + (long long)(unsigned)(wide(al, bl) >> 31);
    return (wide(ah, bh) << K) + (c >> (31 - K));
}

// product with the scale S (S <= SA + SB; the result must fit)
template <int S, int SA, int SB>
__device__ __forceinline__ Fx<S> mul(Fx<SA> a, Fx<SB> b)
{
    constexpr int K = SA + SB - S;
    static_assert(K >= 0 && K < 31, "a product keeps at most 30 extra bits");
    if (K == 0) return {mul62(a.v, b.v)};
    return {mul62k<K>(a.v, b.v)};
}

// the same number with another scale (a larger one drops low bits, a smaller
// one must still hold it)
template <int S, int SA>
__device__ __forceinline__ Fx<S> to(Fx<SA> a)
{
    if (S >= SA) return {a.v >> (S >= SA ? S - SA : 0)};
    return {a.v << (S < SA ? SA - S : 0)};
}
template <int S>
__device__ __forceinline__ Fx<S> operator+(Fx<S> a, Fx<S> b) { return {a.v + b.v}; }
template <int S>
__device__ __forceinline__ Fx<S> operator-(Fx<S> a, Fx<S> b) { return {a.v - b.v}; }
template <int S>
__device__ __forceinline__ Fx<S> operator-(Fx<S> a) { return {-a.v}; }
template <int S>
__device__ __forceinline__ Fx<S> abs_of(Fx<S> a)
{
    const long long m = a.v >> 63;
    return {(a.v ^ m) - m};
}
__device__ __forceinline__ int hi_word(long long v) { return (int)(v >> 32); }

// |x| >= 2^(S - LOG) (on the high word: to 2^-30 of the scale)
template <int LOG, int S>
__device__ __forceinline__ bool outside(Fx<S> a)
{
    return (unsigned)(hi_word(a.v) + (1 << (30 - LOG))) >= (unsigned)(2 << (30 - LOG));
}

// x in [2^(S - L) (1 + 2^(L - 30)), 2^S), on the high word.  The lower end is left
// out: its reciprocal (or reciprocal root) is a power of two that does not fit the
// 62 bits, and its high limb would wrap to the negative number.
template <int L, int S>
__device__ __forceinline__ bool in_window(Fx<S> a)
{
    constexpr unsigned lo = (1u << (30 - L)) + 1;
    return (unsigned)hi_word(a.v) - lo < (1u << 30) - lo;
}

// the number rounded to 53 significant bits (ties upwards), as binary64 holds it
template <int S>
__device__ __forceinline__ Fx<S> round53(Fx<S> a)
{
    int top;   // position of the highest bit that differs from the sign, in the high word
    asm("bfind.s32 %0, %1;" : "=r"(top) : "r"(hi_word(a.v)));
    const unsigned one = 1u << max(top - 20, 0);
    const unsigned long long r = (unsigned long long)a.v + (one >> 1);
    return {(long long)((r & 0xffffffff00000000ull) | ((unsigned)r & (0u - one)))};
}

// z = 1/sqrt(x) as Fx<L/2> and s = sqrt(x) as Fx<0> for x in (2^-L, 1) as in_window
// admits it, L = 6 or 8: the hardware's binary32 estimate z0 (relative error about
// 2^-22) and one third-order step, with e = 1 - x z0^2: z = z0 (1 + e/2 + 3 e^2/8)
// (Householder's method), error O(e^3) below the last bit.  z0 has FB fraction
// bits (exact: its mantissa has 24 bits and z0 >= 1).
template <int L>
__device__ __forceinline__ void rsqrt_sqrt(Fx<0> x, Fx<L / 2> &z, Fx<0> &s)
{
    constexpr int FB = 30 - L / 2;
    const float xf = __int_as_float(__float_as_int(__int2float_rn(limb_hi(x.v))) - (31 << 23));
    float zf;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(zf) : "f"(xf));
    const int z0 = __float2int_rn(zf * (float)(1 << FB));
    // t = x z0 (62 fraction bits), then 1 - t z0
    const int xh = limb_hi(x.v), xl = limb_lo(x.v);
    const long long t = (wide(xh, z0) << (31 - FB)) + (wide(xl, z0) >> FB);
    const int th = limb_hi(t), tl = limb_lo(t);
    const long long p = (wide(th, z0) << (31 - FB)) + (wide(tl, z0) >> FB);
    const long long e = kOne62 - p;   // |e| < 2^42
    const int es = (int)(e >> 20);
    const int e2 = (int)(wide(es, es) >> 22);               // e^2, 62 fraction bits
    const long long h = (e >> 1) + ((3 * e2) >> 3);
    const int hh = limb_hi(h), hl = limb_lo(h);
    z.v = ((long long)z0 << 32) + (wide(z0, hh) << 1) + (wide(z0, hl) >> 30);
    s.v = t + wide(th, hh) + ((wide(th, hl) + wide(tl, hh)) >> 31);
}

// 1/x as Fx<0> for x in [5/4, 3]: binary32 estimate (31 fraction bits) and one
// third-order Newton step, 1/x = r0 (1 + e + e^2), e = 1 - x r0
__device__ __forceinline__ Fx<0> rcp_above1(Fx<4> x)
{
    float rf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(__int2float_rn(limb_hi(x.v))));   // x 2^27
    const int r0 = __float2int_rn(rf * 288230376151711744.0f);                             // 2^58
    const int xh = limb_hi(x.v), xl = limb_lo(x.v);
    const long long p = (wide(xh, r0) << 4) + (wide(xl, r0) >> 27);
    const long long e = kOne62 - p;
    const int es = (int)(e >> 20);
    const long long h = e + (long long)(int)(wide(es, es) >> 22);
    const int hh = limb_hi(h), hl = limb_lo(h);
    return {((long long)r0 << 31) + wide(r0, hh) + (wide(r0, hl) >> 31)};
}

// 1/x as Fx<L> for x in (2^-L, 1) as in_window admits it, in the same way (30 - L fraction bits of the estimate)
template <int L>
__device__ __forceinline__ Fx<L> rcp_below1(Fx<0> x)
{
    constexpr int FB = 30 - L;
    const int xh = limb_hi(x.v), xl = limb_lo(x.v);
    float rf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(__int2float_rn(xh)));   // x 2^31
    const int r0 = __float2int_rn(rf * (2147483648.0f * (float)(1 << FB)));
    const long long p = (wide(xh, r0) << (31 - FB)) + (wide(xl, r0) >> FB);
    const long long e = kOne62 - p;
    const int es = (int)(e >> 20);
    const long long h = e + (long long)(int)(wide(es, es) >> 22);
    const int hh = limb_hi(h), hl = limb_lo(h);
    return {((long long)r0 << 32) + (wide(r0, hh) << 1) + (wide(r0, hl) >> 30)};
}

}  // namespace fx
}  // namespace rok
