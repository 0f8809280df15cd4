// Wide fixed-point numbers for the FP64 operator products.
//
// GB300 issues FP64 at 2 lanes per clock and SM, 32-bit multiply-add with a
// 64-bit sum (IMAD.WIDE) at 64 and 32-bit add at 128 (measured: 1.9, 60 and
// 120), so a product sum of the precision of FP64 is several times cheaper in
// integers.  A value is l2 2^52 + l1 2^26 + l0 with 32-bit limbs that carry 26
// bits each and leave the rest of the word for sums: additions are three
// independent 32-bit adds without carries, products are taken limb by limb into
// 64-bit sums and carried once per result.
//   - inputs: |value| < 2^75 (gm_fx_from_double), i.e. 75 bits below the power
//     of two at or above the largest input of the tile;
//   - 8-point transforms and sums of up to 28 (signed limbs: 36) results fit the words;
//   - coefficients: |c| < 1 as c2 2^-26 + c1 2^-52 + c0 2^-78, exact for the
//     53 bits of a double within 2^25 of the largest (moduli: within 2^21; the
//     entries of K_b to 2^-83 of the largest row sum, so that those of flat cells,
//     a^2 apart at an aspect ratio a, keep their bits);
//   - a product sum loses at most about 2^3 units of the last place (the limb
//     pairs below it), a node of the operators about 2^6, so results are exact
//     to 2^-69 of the tile's largest term, 16 bits below FP64's rounding.
#pragma once

#include <stdint.h>
#include <string.h>

constexpr int GM_FX_RADIX = 26;
constexpr int GM_FX_MASK = (1 << GM_FX_RADIX) - 1;
constexpr int GM_FX_IN = 75;       // bits of an input value
constexpr int GM_FX_GRADE = 16;    // bits of grading inside a tile beyond which fixed point is not tried

__host__ __device__ inline int64_t gm_fx_bits(double x)
{
    int64_t b;
    memcpy(&b, &x, 8);
    return b;
}
__host__ __device__ inline double gm_fx_real(int64_t b)
{
    double x;
    memcpy(&x, &b, 8);
    return x;
}

// limbs of x / 2^(ex - 75) rounded towards zero, for |x| < 2^ex (biased
// exponent field of 2^(ex - 1) given as top); smaller than one unit gives 0.
// x must be finite; subnormal x gives 0 (top is far above them).
__host__ __device__ inline void gm_fx_from_double(double x, int top, int (&l)[3])
{
    const int64_t b = gm_fx_bits(x);
    const int e = (int)((uint64_t)b >> 52) & 0x7ff;
    const uint64_t m = e ? (((uint64_t)b & 0xfffffffffffffull) | 0x10000000000000ull) : 0ull;
    // m holds 53 bits; value = m 2^(75 - 53 - d), d = top - e >= 0
    int d = top - e;
    if (d > 90) d = 90;
    const uint64_t M = m << 11;                    // top bit at 63: the value is M 2^(11 - d)
    // limb 2: value >> 52 = M >> (41 + d); limb 1: bits 26..51 = M >> (15 + d); limb 0: M << 11 >> d
    const int s2 = 41 + d, s1 = 15 + d;
    const int h2 = s2 < 64 ? (int)(M >> s2) : 0;
    const int h1 = s1 < 64 ? (int)(M >> s1) & GM_FX_MASK : 0;
    const int s0 = d - 11;
    const int h0 = (s0 >= 64 ? 0 : s0 >= 0 ? (int)(M >> s0) : (int)(M << -s0)) & GM_FX_MASK;
    const int sg = (int)(b >> 63);
    l[0] = (h0 ^ sg) - sg;
    l[1] = (h1 ^ sg) - sg;
    l[2] = (h2 ^ sg) - sg;
}

// limbs of a coefficient 0 <= c < 1 in 78 bits; top is the biased exponent of the
// largest coefficient's power of two (c's own exponent field is at most top)
__host__ __device__ inline void gm_fx_coef(double c, int top, int (&l)[3])
{
    const int64_t b = gm_fx_bits(c);
    const int e = (int)((uint64_t)b >> 52) & 0x7ff;
    const uint64_t m = e ? (((uint64_t)b & 0xfffffffffffffull) | 0x10000000000000ull) : 0ull;
    int d = top - e;                               // c = m 2^(78 - 53 - d) units of 2^-78
    const uint64_t M = d < 78 ? m << 11 : 0;       // 78 bits: M 2^(14 - d)
    if (d > 77) d = 77;
    const int s2 = 38 + d, s1 = 12 + d, s0 = d - 14;
    l[2] = s2 < 64 ? (int)(M >> s2) : 0;
    l[1] = s1 < 64 ? (int)(M >> s1) & GM_FX_MASK : 0;
    l[0] = (s0 >= 0 ? (int)(M >> s0) : (int)(M << -s0)) & GM_FX_MASK;
}

// limbs of a coefficient 0 <= c < 1 as l2 2^-22 + l1 2^-48 + l0 2^-74
__host__ __device__ inline void gm_fx_coef22(double c, int top, int (&l)[3])
{
    const int64_t b = gm_fx_bits(c);
    const int e = (int)((uint64_t)b >> 52) & 0x7ff;
    const uint64_t m = e ? (((uint64_t)b & 0xfffffffffffffull) | 0x10000000000000ull) : 0ull;
    int d = top - e;                               // c = m 2^(74 - 53 - d) units of 2^-74
    const uint64_t M = d < 74 ? m << 11 : 0;       // 74 bits: M 2^(10 - d)
    if (d > 73) d = 73;
    const int s2 = 42 + d, s1 = 16 + d, s0 = d - 10;
    l[2] = s2 < 64 ? (int)(M >> s2) : 0;
    l[1] = s1 < 64 ? (int)(M >> s1) & GM_FX_MASK : 0;
    l[0] = (s0 >= 0 ? (int)(M >> s0) : (int)(M << -s0)) & GM_FX_MASK;
}

// sums of limb products of one result, by weight
struct FxAcc {
    int64_t a2, a1, a0;
};
__host__ __device__ inline void gm_fx_mac(FxAcc& s, const int (&x)[3], int c2, int c1, int c0)
{
    s.a2 += (int64_t)x[2] * c2;
    s.a1 += (int64_t)x[1] * c2;
    s.a1 += (int64_t)x[2] * c1;
    s.a0 += (int64_t)x[0] * c2;
    s.a0 += (int64_t)x[1] * c1;
    s.a0 += (int64_t)x[2] * c0;
}
// The same with a coefficient c2 2^-30 + c1 2^-56 (|c2| <= 2^30).  Sums and
// carried limbs then weigh 2^4 less: (2^48, 2^22, 2^-4); multiplied by a coefficient
// whose top limb has 22 bits (gm_fx_coef22) they are back at (2^52, 2^26, 1).
__host__ __device__ inline void gm_fx_mac2(FxAcc& s, const int (&x)[3], int c2, int c1)
{
    s.a2 += (int64_t)x[2] * c2;
    s.a1 += (int64_t)x[1] * c2;
    s.a1 += (int64_t)x[2] * c1;
    s.a0 += (int64_t)x[0] * c2;
    s.a0 += (int64_t)x[1] * c1;
}
// and with a third limb c0 2^-82 below (|c1|, |c0| <= 2^25): a product loses 2^-1
// units, the carried sum 2^-3
__host__ __device__ inline void gm_fx_mac3(FxAcc& s, const int (&x)[3], int c2, int c1, int c0)
{
    gm_fx_mac2(s, x, c2, c1);
    s.a0 += (int64_t)x[2] * c0;
}

// carried limbs: l0, l1 in [0, 2^26), l2 signed
__host__ __device__ inline void gm_fx_carry(const FxAcc& s, int (&l)[3])
{
    const int64_t t0 = s.a1 + (s.a0 >> GM_FX_RADIX);
    l[0] = (int)t0 & GM_FX_MASK;
    const int64_t t1 = s.a2 + (t0 >> GM_FX_RADIX);
    l[1] = (int)t1 & GM_FX_MASK;
    l[2] = (int)(t1 >> GM_FX_RADIX);
}
// the same with l0, l1 in [-2^25, 2^25)
__host__ __device__ inline void gm_fx_carry_signed(const FxAcc& s, int (&l)[3])
{
    constexpr int H = 1 << (GM_FX_RADIX - 1);
    const int64_t t0 = s.a1 + (s.a0 >> GM_FX_RADIX) + H;
    l[0] = ((int)t0 & GM_FX_MASK) - H;
    const int64_t t1 = s.a2 + (t0 >> GM_FX_RADIX) + H;
    l[1] = ((int)t1 & GM_FX_MASK) - H;
    l[2] = (int)(t1 >> GM_FX_RADIX);
}

// Product sums with one limb more below (weight 2^-26), for results whose terms
// carry coefficients far apart: l[0] is that limb, l[1..3] those above.
struct FxAcc4 {
    int64_t a2, a1, a0, am;
};
__host__ __device__ inline void gm_fx_mac4(FxAcc4& s, const int (&x)[3], int c2, int c1, int c0)
{
    s.a2 += (int64_t)x[2] * c2;
    s.a1 += (int64_t)x[1] * c2;
    s.a1 += (int64_t)x[2] * c1;
    s.a0 += (int64_t)x[0] * c2;
    s.a0 += (int64_t)x[1] * c1;
    s.a0 += (int64_t)x[2] * c0;
    s.am += (int64_t)x[0] * c1;
    s.am += (int64_t)x[1] * c0;
}
__host__ __device__ inline void gm_fx_carry4_signed(const FxAcc4& s, int (&l)[4])
{
    constexpr int H = 1 << (GM_FX_RADIX - 1);
    const int64_t tm = s.a0 + (s.am >> GM_FX_RADIX) + H;
    l[0] = ((int)tm & GM_FX_MASK) - H;
    const int64_t t0 = s.a1 + (tm >> GM_FX_RADIX) + H;
    l[1] = ((int)t0 & GM_FX_MASK) - H;
    const int64_t t1 = s.a2 + (t0 >> GM_FX_RADIX) + H;
    l[2] = ((int)t1 & GM_FX_MASK) - H;
    l[3] = (int)(t1 >> GM_FX_RADIX);
}

// nearest double of l2 2^52 + l1 2^26 + l0 (one rounding): the bits below 2^52
// and the rest are exact doubles, joined by one fused multiply-add
__host__ __device__ inline double gm_fx_to_double(int l0, int l1, int l2)
{
    const int64_t t = (int64_t)l1 * (1 << GM_FX_RADIX) + l0;
    const int hi = l2 + (int)(t >> 52);
    const double lo = gm_fx_real((t & 0xfffffffffffffll) | 0x4330000000000000ll) - 4503599627370496.0;
    const double dh = gm_fx_real((int64_t)(0x4330000000000000ull | (uint32_t)(hi ^ 0x80000000))) - 4503601774854144.0;
    return fma(dh, 4503599627370496.0, lo);
}

// double of l3 2^52 + l2 2^26 + l1 + l0 2^-26, within one unit of its last place:
// the middle part is kept in [-2^51, 2^51), so that values of either sign below
// one unit keep their lowest limb
__host__ __device__ inline double gm_fx_to_double4(int l0, int l1, int l2, int l3)
{
    const int64_t t = (int64_t)l2 * (1 << GM_FX_RADIX) + l1;
    const int64_t up = (t + (1ll << 51)) >> 52;
    const int hi = l3 + (int)up;
    const double mid = gm_fx_real((int64_t)(0x4338000000000000ull + (uint64_t)(t - up * (1ll << 52)))) - 6755399441055744.0;
    const double dl = gm_fx_real((int64_t)(0x4330000000000000ull | (uint32_t)(l0 ^ 0x80000000))) - 4503601774854144.0;
    const double dh = gm_fx_real((int64_t)(0x4330000000000000ull | (uint32_t)(hi ^ 0x80000000))) - 4503601774854144.0;
    return fma(dh, 4503599627370496.0, fma(dl, 1.4901161193847656e-08, mid));
}
