// Packed pairs of floats: two IEEE operations per instruction.  A packed product
// whose only use is a packed sum is contracted with it by the compiler, so where
// both roundings count the product goes through fma with -0 (the sums below) or
// the sum is taken one float at a time (add2).
#pragma once

namespace csc {

__device__ __forceinline__ unsigned long long pack2(float lo, float hi)
{
    unsigned long long x;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(lo), "f"(hi));
    return x;
}
__device__ __forceinline__ void unpack2(unsigned long long x, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b,
                                                   unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    float a0, a1, b0, b1;
    unpack2(a, a0, a1);
    unpack2(b, b0, b1);
    return pack2(__fadd_rn(a0, b0), __fadd_rn(a1, b1));
}
constexpr unsigned long long kOne2 = 0x3f8000003f800000ull;
constexpr unsigned long long kMinusOne2 = 0xbf800000bf800000ull;
constexpr unsigned long long kMinusZero2 = 0x8000000080000000ull;

// df_add_prod on two accumulators at once, negated: (hi, lo) -= a b; nb = -b.
// (The rounded product enters TwoSum as a nb, the one form that is needed.)
__device__ __forceinline__ void df2_sub_prod(unsigned long long &hi, unsigned long long &lo,
                                             unsigned long long a, unsigned long long b,
                                             unsigned long long nb)
{
    const unsigned long long np = fma2(a, nb, kMinusZero2);
    const unsigned long long pe = fma2(a, b, np);                   // a b - p
    const unsigned long long s = fma2(hi, kOne2, np);
    const unsigned long long bv = fma2(hi, kMinusOne2, s);          // s - hi
    const unsigned long long t1 = fma2(bv, kMinusOne2, s);          // s - bv
    const unsigned long long t2 = fma2(t1, kMinusOne2, hi);         // hi - (s - bv)
    const unsigned long long t3 = fma2(bv, kMinusOne2, np);         // np - bv
    const unsigned long long e = fma2(pe, kMinusOne2, fma2(t2, kOne2, t3));
    hi = s;
    lo = fma2(lo, kOne2, e);
}

}  // namespace csc
