// Dot products of binary64 entries on the integer pipe (FMA build).
//
// Gram-Schmidt needs two FP64 multiply-adds for every basis entry it reads (a
// projection and an update), and GB300 issues FP64 at 2 lane-operations per SM
// and clock.  Here a thread's part of a projection is summed in integers, which
// overlaps the FP64 update: the entries of each operand (at most 16) become
// fixed-point numbers below 2^57 in units set by the operand's largest exponent,
// and the products of their 29-bit limbs are accumulated exactly.  One rounding
// to 2^-56 of the largest product and the conversion to binary64 end the sum;
// the entries themselves lose (towards zero) what lies below 2^-57 of the largest one of
// the thread.  So the error is below 2^-52 of (largest |v|) (largest |w|) for 8 terms:
// smaller than that of a chain of binary64 multiply-adds where the thread's entries
// are of similar size, as neighbouring cells' are, but relative to the largest
// product, not to each: a sum whose large entries of one vector all meet small ones
// of the other keeps fewer digits of its own.  An entry
// costs 16 integer instructions an operand and four 32 x 32 -> 64 multiply-adds
// (8 to 10 SM clocks a warp together, against 16 for one FP64 instruction).
// Operands that are zero, non-finite or far outside the usual exponents are left
// to the caller's binary64 sum.
#pragma once
#include <cuda_runtime.h>

namespace rok {
namespace idot {

constexpr int kMaxTerms = 16;   // |cross terms| <= 16 * 2 * 2^28 * 2^29 = 2^62

struct Limb {
    int h, l;   // x = h 2^29 + l, |h| <= 2^28, 0 <= l < 2^29
};
struct Acc {
    long long hi, mid, lo;
};

__device__ __forceinline__ int magnitude(double x) { return __double2hiint(x) & 0x7fffffff; }
// exponent field of the largest of the magnitudes (high words) seen
__device__ __forceinline__ int top(int mag) { return mag & 0x7ff00000; }
// the product of two such units stays a normal binary64 number
__device__ __forceinline__ bool usable(int t) { return (unsigned)(t - (600 << 20)) < (unsigned)(846 << 20); }

// x in units of 2^(t - 1079), t the exponent field `top' of its operand
// (truncated towards zero; subnormals are below the unit)
__device__ __forceinline__ Limb limbs(double x, int t)
{
    const int hi = __double2hiint(x);
    const unsigned n = (unsigned)(t - (hi & 0x7ff00000)) >> 20;
    const unsigned long long m =
        ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32 | (unsigned)__double2loint(x)) << 4;
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(n));   // 64 and more: zero
    const long long s = (long long)(hi >> 31);
    const long long v = ((long long)r ^ s) - s;
    return {(int)(v >> 29), (int)v & 0x1fffffff};
}

__device__ __forceinline__ void mad(Acc &a, Limb x, Limb y)
{
    a.hi += (long long)x.h * y.h;
    a.mid += (long long)x.h * y.l;
    a.mid += (long long)x.l * y.h;
    a.lo += (long long)x.l * y.l;
}

// the sum as binary64; ta, tb the operands' exponent fields
__device__ __forceinline__ double finish(const Acc &a, int ta, int tb)
{
    const long long s = a.hi + ((a.mid + (a.lo >> 29) + (1ll << 28)) >> 29);   // units of 2^(ta + tb - 2100)
    const double d = (double)s;
    const int up = (int)((unsigned)ta + (unsigned)tb - (2100u << 20));
    return __hiloint2double(s != 0 ? __double2hiint(d) + up : 0, __double2loint(d));
}

}  // namespace idot
}  // namespace rok
