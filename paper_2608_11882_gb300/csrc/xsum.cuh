// The exact-sum FP64 arithmetic shared by the heat and CG kernels: values of
// an FP64 vector become 64-bit fixed-point integers on the vector's current
// scale, sums of them are exact, and a sum returns to FP64 with one rounding.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace hcg {

// Each value u of an FP64 vector (a heat field, a CG direction) becomes a
// signed integer U within two units of u 2^(1080 - e), where e is the largest
// biased exponent field among the vector's values (so |U| <= 2^58; values more
// than 58 binades below the maximum become 0 or -1).  A stencil sum of such
// integers -- the heat numerator L = S - 6U, the Laplacian 6U - S -- is then
// exact in 64 bits (|L| < 12 2^58 + 12), and is rounded once to the nearest
// double L 2^(e - 1080).  Against the same sum in exact arithmetic the error
// is below 24 2^-57 max|u| plus that one rounding.  GB300 runs FP64 <-> int64
// conversion instructions at its narrow FP64 rate, so U is formed with integer
// instructions; L becomes a double either with integer instructions
// (xs_unfix) or with one FP64-pipe conversion followed by an exact scaling --
// the same double either way, so kernels may mix the two to balance pipes.
// The caller tracks e (non-negative doubles order like their bit patterns, so
// the largest |u| bit pattern gives it) and keeps vectors whose e lies outside
// [xs_emax_lo, kXsEmaxHi] -- zero or tiny vectors, values near overflow, NaN,
// Inf -- on the FP64 pipe, which also carries NaN and Inf through.
constexpr int kXsEmaxLo = 70, kXsEmaxHi = 2040;

// Smallest e for which L 2^(e - 1080) (|L| >= 1) and r 2^(e - 1080) are normal.
__device__ __forceinline__ int xs_emax_lo(double r)
{
    const int er = (int)((unsigned long long)__double_as_longlong(r) >> 52) & 0x7ff;
    return er == 0 ? kXsEmaxLo : max(kXsEmaxLo, 1081 - er);
}

__device__ __forceinline__ bool xs_native(int emax, double r)
{
    return emax < xs_emax_lo(r) || emax > kXsEmaxHi;
}

// r 2^(e - 1080), exact when e >= xs_emax_lo(r).
__device__ __forceinline__ double xs_r2(double r, int emax)
{
    return r * __longlong_as_double((long long)(emax - 57) << 52);
}

// The fixed-point integer of the double with bit pattern `bits` (its exponent
// field must not exceed emax): the mantissa with its implicit bit, times 2^SH,
// in ones' complement for negative values, shifted right arithmetically by
// emax - e -- floor((u 2^(1075 + SH - emax)) - [u < 0] 2^-t), within two units
// of u 2^(1075 + SH - emax).  Zeros and subnormals give 0 or -1 for emax >= 64.
//
// The kernels that convert are bound by the integer pipe, so the two
// conversions count instructions: PTX's shifts clamp amounts above 63, which
// C++'s do not, so no minimum or mask is taken; emax - e is one subtraction and
// one shift (the ones below emax's field keep the mantissa from borrowing); and
// xs_unfix selects only the high word for a zero.  512^3 FP64 heat 393.6 ->
// 384.9 us per step, 64 requests of 256^3 31.2 -> 30.9 ms, variable kappa at
// 510^3 890 -> 856 us.
template <int SH = 5>
__device__ __forceinline__ long long xs_fix(long long bits, int emax)
{
    const unsigned hi = (unsigned)((unsigned long long)bits >> 32), lo = (unsigned)bits;
    const unsigned s = (unsigned)((int)hi >> 31);   // 0 or all ones
    const unsigned t = (((unsigned)emax << 21 | 0x1fffffu) - (hi << 1)) >> 21;   // emax - e
    constexpr unsigned one = 1u << (20 + SH);   // the implicit bit
    const unsigned mh = ((__funnelshift_l(lo, hi, SH) & (one - 1u)) | one) ^ s;
    const unsigned ml = (lo << SH) ^ s;
    long long q;
    asm("shr.s64 %0, %1, %2;" : "=l"(q) : "l"((long long)(((unsigned long long)mh << 32) | ml)), "r"(t));
    return q;
}

// x 2^(emax - 1080) rounded to the nearest double, ties to even (|x| < 2^63: the
// six-point sums stay below 2^62, the variable-coefficient ones below 1.43 2^62;
// xs_emax_lo <= emax <= kXsEmaxHi, so the result is a normal number or zero).
__device__ __forceinline__ double xs_unfix(long long x, int emax)
{
    const unsigned long long s = (unsigned long long)(x >> 63);
    const unsigned long long a = ((unsigned long long)x ^ s) - s;
    const int lz = __clzll((long long)a);                       // >= 1; 64 for a = 0
    unsigned long long n;                                       // leading one at bit 62
    asm("shl.b64 %0, %1, %2;" : "=l"(n) : "l"(a), "r"(lz - 1));
    const unsigned long long q = (n + 0x1ffull + ((n >> 10) & 1ull)) >> 10;   // 2^52 <= q <= 2^53, or 0
    // biased exponent emax + 6 - lz; q's bit 52 (or a carry to 53) adds into the exponent field
    const unsigned hi = (unsigned)(q >> 32) + ((unsigned)(emax + 5 - lz) << 20) +
                        ((unsigned)s & 0x80000000u);
    return __longlong_as_double((long long)(((unsigned long long)(a ? hi : 0u) << 32) | (unsigned)q));
}

// The same double as xs_unfix, through one FP64-pipe conversion (rounding to
// nearest even) and an exact adjustment of the exponent field.
__device__ __forceinline__ double xs_unfix_dp(long long x, int emax)
{
    const long long b = __double_as_longlong(__ll2double_rn(x));
    return x ? __longlong_as_double(b + (long long)(emax - 1080) * (1ll << 52)) : 0.0;
}

// L = S - 6U of a point from its seven fixed-point values.
__device__ __forceinline__ long long xs_numerator(long long c, long long xm, long long xp, long long ym,
                                                  long long yp, long long zm, long long zp)
{
    return ((xm + xp) + (ym + yp)) + (zm + zp) - 6 * c;
}

// u' = fma(r, L 2^(emax - 1080), uc): DPCONV converts L on the FP64 pipe and
// scales r instead (r2 = xs_r2(r, emax)); both round the same exact product.
template <bool DPCONV>
__device__ __forceinline__ double xs_apply(double uc, long long L, double r, double r2, int emax)
{
    if constexpr (DPCONV) return __fma_rn(r2, __ll2double_rn(L), uc);
    return __fma_rn(r, xs_unfix(L, emax), uc);
}

// ---- weighted differences -------------------------------------------------
// d w / 2^64 to within 2.5 units, w = hi 2^32 + lo with a signed low part and
// 0 <= hi < 2^31: the three 32-bit products that reach the high word.
__device__ __forceinline__ long long xs_mulhi3(long long d, int hi, int lo)
{
    const int dh = (int)(d >> 32);
    return (long long)dh * hi + __mulhi(dh, lo) + (long long)__umulhi((unsigned)d, (unsigned)hi);
}

// The flux c d through a face: d the difference of two values' integers with
// SH = 7 (|d| < 2^61, so units of u 2^(1082 - emax)), c in [1, 2) the sum of two
// coefficients in [0.5, 1), given as their bit patterns.  Returns c d / 4 to
// within 2.5 units, c as the 63-bit integer c 2^62 (exact: the sum of the two
// 53-bit significands, shifted).  Six of them sum without overflow (below
// 6 1.9/4 2^61), in units of u 2^(1080 - emax).
__device__ __forceinline__ long long xs_flux(long long ca, long long cb, long long d)
{
    const unsigned long long s = (unsigned long long)(ca + cb) << 9;   // bits 0..52 of the sum, the exponents above
    const int lo = (int)(unsigned)s;
    const int hi = (int)(((unsigned)(s >> 32) & 0x3fffffffu) | 0x40000000u) + (int)((unsigned)lo >> 31);
    return xs_mulhi3(d, hi, lo);
}

// |u| of a result as the high word of its bit pattern (the exponent field and
// the top of the mantissa): what the per-step maximum needs.
__device__ __forceinline__ unsigned xs_abs_hi(double v)
{
    return (unsigned)((unsigned long long)__double_as_longlong(v) >> 32) & 0x7fffffffu;
}


}  // namespace hcg
