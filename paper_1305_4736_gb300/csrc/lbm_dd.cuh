// lbm_dd.cuh -- double-float arithmetic for the float64 mode on the float32 pipe.
//
// GB300 issues float32 FMAs at 128 lanes per SM cycle and float64 ones at about 1.7, so the
// float64 mode's step can run faster in double-float arithmetic: a value is an unevaluated sum
// hi + lo of two float32 numbers (48 significand bits), and each operation is built from
// error-free transformations on the float32 pipe (Dekker, "A floating-point technique for
// extending the available precision", Numer. Math. 18, 1971; Knuth, TAOCP vol. 2, 4.2.2:
// TwoSum; Fast2Sum; the product error from an FMA).  Relative rounding of an operation is
// about 2^-47, against 2^-53 in float64.
//
// Values are kept unnormalised between operations: a sum or product returns the high part and
// its exact error plus the low parts, without the final Fast2Sum that would make
// |lo| <= ulp(hi) / 2.  The pair still holds the value to the same accuracy (lo stays within a
// few units of 2^-24 of the operands' magnitudes), and every operation here reads both parts,
// so only the places that look at hi alone renormalise first: the MC slope's comparisons and
// sign test, and the reciprocal's Newton step.  The populations stay float64 in HBM: a staged
// value is split into hi + lo (rounded to nearest) with integer operations, since
// float32 <-> float64 conversions run at the float64 rate on this part and the split is a phase
// of its own; an updated value is rounded back to float64 by one float64 addition, which runs
// beside the float32 arithmetic of the other warps.
//
// Every float32 operation here uses the _rn intrinsics, which the compiler neither contracts
// into FMAs nor reorders, so the transformations stay error-free.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

struct dd {
    float hi, lo;
};

// Host: the double-float value nearest to x (hi = x rounded to float, lo = the rest rounded).
inline dd dd_host(double x)
{
    const float h = (float)x;
    return dd{h, (float)(x - (double)h)};
}

__device__ __forceinline__ dd ddf(float h) { return dd{h, 0.0f}; }

// Fast2Sum (|a| >= |b| or a == 0): s + e = a + b exactly.
__device__ __forceinline__ dd fast2sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return dd{s, __fsub_rn(b, __fsub_rn(s, a))};
}

// a + b: TwoSum of the high parts, the low parts added to its error (8 operations).
__device__ __forceinline__ dd operator+(dd a, dd b)
{
    const float s = __fadd_rn(a.hi, b.hi);
    const float v = __fsub_rn(s, a.hi);
    const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, v)), __fsub_rn(b.hi, v));
    return dd{s, __fadd_rn(e, __fadd_rn(a.lo, b.lo))};
}

__device__ __forceinline__ dd operator-(dd a) { return dd{-a.hi, -a.lo}; }

__device__ __forceinline__ dd operator-(dd a, dd b)
{
    const float s = __fsub_rn(a.hi, b.hi);
    const float v = __fsub_rn(s, a.hi);
    const float e = __fsub_rn(__fsub_rn(a.hi, __fsub_rn(s, v)), __fadd_rn(b.hi, v));
    return dd{s, __fadd_rn(e, __fsub_rn(a.lo, b.lo))};
}

// a * b: the product of the high parts and its exact error (from an FMA) plus the cross
// terms (4 operations).
__device__ __forceinline__ dd operator*(dd a, dd b)
{
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    return dd{p, e};
}

// a * c for a float32 constant c (3).
__device__ __forceinline__ dd operator*(dd a, float c)
{
    const float p = __fmul_rn(a.hi, c);
    float e = __fmaf_rn(a.hi, c, -p);
    e = __fmaf_rn(a.lo, c, e);
    return dd{p, e};
}
__device__ __forceinline__ dd operator*(float c, dd a) { return a * c; }

// a * 2^k (exact).
__device__ __forceinline__ dd scale2(dd a, float p2) { return dd{__fmul_rn(a.hi, p2), __fmul_rn(a.lo, p2)}; }

// a * b + c (12).
__device__ __forceinline__ dd fma_dd(dd a, dd b, dd c)
{
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    const float s = __fadd_rn(p, c.hi);
    const float v = __fsub_rn(s, p);
    const float t = __fadd_rn(__fsub_rn(p, __fsub_rn(s, v)), __fsub_rn(c.hi, v));
    return dd{s, __fadd_rn(t, __fadd_rn(e, c.lo))};
}

// 1/x: the float32 approximate reciprocal y of x rounded to float (relative error below
// 2^-22), then one Newton step y + y (1 - x y) with 1 - x y formed in double-float and its two
// parts summed (the residual's high part alone can be of the size of its low part); relative
// error about 2^-44.
__device__ __forceinline__ dd recip(dd x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__fadd_rn(x.hi, x.lo)));
    const dd r = ddf(1.0f) - x * y;
    return fast2sum(y, __fmul_rn(y, __fadd_rn(r.hi, r.lo)));
}

// ---------------------------------------------------------------------------
// Pairs of double-float values, (q, q + 4) of the population pairs: hi and lo parts as float2
// for the f32x2 instructions.  A packed instruction does the work of two at half the issue
// slots and the same lane rate (measured with chains of independent operations: 122 lane
// operations per cycle per SM packed, 119 scalar), so the double-float chains leave half of the
// issue slots to the loads, selects and shuffles.  Each lane rounds as the scalar operation.
// ---------------------------------------------------------------------------
struct dd2 {
    float2 hi, lo;
};

__device__ __forceinline__ float2 neg2(float2 a) { return f2(-a.x, -a.y); }
__device__ __forceinline__ dd2 pack(dd a, dd b) { return dd2{f2(a.hi, b.hi), f2(a.lo, b.lo)}; }
__device__ __forceinline__ dd2 bcast(dd a) { return pack(a, a); }
__device__ __forceinline__ dd first(dd2 a) { return dd{a.hi.x, a.lo.x}; }
__device__ __forceinline__ dd second(dd2 a) { return dd{a.hi.y, a.lo.y}; }

__device__ __forceinline__ dd2 operator+(dd2 a, dd2 b)
{
    const float2 s = add2(a.hi, b.hi);
    const float2 v = sub2(s, a.hi);
    const float2 e = add2(sub2(a.hi, sub2(s, v)), sub2(b.hi, v));
    return dd2{s, add2(e, add2(a.lo, b.lo))};
}

__device__ __forceinline__ dd2 operator-(dd2 a, dd2 b)
{
    const float2 s = sub2(a.hi, b.hi);
    const float2 v = sub2(s, a.hi);
    const float2 e = sub2(sub2(a.hi, sub2(s, v)), add2(b.hi, v));
    return dd2{s, add2(e, sub2(a.lo, b.lo))};
}

__device__ __forceinline__ dd2 operator*(dd2 a, dd2 b)
{
    const float2 p = mul2(a.hi, b.hi);
    float2 e = fma2(a.hi, b.hi, neg2(p));
    e = fma2(a.hi, b.lo, e);
    e = fma2(a.lo, b.hi, e);
    return dd2{p, e};
}

// by float32 constants, one per lane (3 packed operations)
__device__ __forceinline__ dd2 operator*(dd2 a, float2 c)
{
    const float2 p = mul2(a.hi, c);
    float2 e = fma2(a.hi, c, neg2(p));
    e = fma2(a.lo, c, e);
    return dd2{p, e};
}

__device__ __forceinline__ dd2 scale2(dd2 a, float p2) { return dd2{mul2(a.hi, f2(p2, p2)), mul2(a.lo, f2(p2, p2))}; }

// The pairs renormalised: |lo| <= ulp(hi) / 2 (Fast2Sum; with a low part larger than the high
// part, after a cancellation, it still returns the pair's value to within 2^-24 of that low part,
// far below the pair's own accuracy).
__device__ __forceinline__ dd2 norm(dd2 a)
{
    const float2 s = add2(a.hi, a.lo);
    return dd2{s, sub2(a.lo, sub2(s, a.hi))};
}

// The first (second) lanes of two pairs.
__device__ __forceinline__ dd2 firsts(dd2 a, dd2 b) { return pack(first(a), first(b)); }
__device__ __forceinline__ dd2 seconds(dd2 a, dd2 b) { return pack(second(a), second(b)); }

// The sum of a pair's two lanes.
__device__ __forceinline__ dd sum_lanes(dd2 a) { return first(a) + second(a); }

// a + b where |b| <= |a| lane by lane (up to a few units in the last place of b): Fast2Sum of the
// high parts, whose error is then exact as TwoSum's is, so the result is that of a + b bit for bit
// (5 packed operations instead of 8).
__device__ __forceinline__ dd2 add_smaller(dd2 a, dd2 b)
{
    const float2 s = add2(a.hi, b.hi);
    return dd2{s, add2(sub2(b.hi, sub2(s, a.hi)), add2(a.lo, b.lo))};
}

// Twice the MC slope, 2 minmod(2a, (a + b)/2, 2b) = sign(a) min(4|a|, 4|b|, |a + b|) when a and
// b agree in sign and 0 otherwise (Sec. III, reading A6); as mc2 of lbm_device.cuh.  a and b
// must be normalised (norm), so that their high parts carry their signs; they agree when
// a.hi b.hi > 0 (a product below 2^-149 counts as disagreement: then the smaller difference
// is below 2^-74, so the slope, at most 4 times it, is below 2^-72, far below the populations'
// 2^-47 resolution, and is taken as 0).  Two candidates x, y of the sign of a are ordered by the float32
// value (x.hi - y.hi) + (x.lo - y.lo), whose sign is that of x - y (zero only for x = y or x, y within
// a few units of 2^-47 of each other, where either is the slope to the pairs' accuracy); the
// smaller magnitude is the lower value for a > 0 and the higher for a < 0, read from the sign of that
// value times a.hi (or s.hi): below 2^-149, where the product reads as zero, the candidates differ by
// less than 2^-74, the flush threshold of the split.  The sum s = a + b is left unnormalised (its low
// part stays within a few units of its high part's last place, which the ordering tolerates where a and b
// agree).  Where they disagree the result is set to zero last: if the high parts cancel, the sign of s.hi
// is not that of s, and no test against s can tell (at an extremum symmetric to 2^-24, s would be taken
// for the slope).  Scaling the candidates by 0 there instead is 1% of the step less, and gives NaN for
// infinities and NaN.
__device__ __forceinline__ dd2 mc2n(dd2 a, dd2 b)
{
    const dd2 s = a + b;
    const float2 ab = mul2(a.hi, b.hi);
    const float2 tab = mul2(add2(sub2(a.hi, b.hi), sub2(a.lo, b.lo)), a.hi);
    dd2 m;
    m.hi.x = tab.x < 0.0f ? a.hi.x : b.hi.x;
    m.lo.x = tab.x < 0.0f ? a.lo.x : b.lo.x;
    m.hi.y = tab.y < 0.0f ? a.hi.y : b.hi.y;
    m.lo.y = tab.y < 0.0f ? a.lo.y : b.lo.y;
    const dd2 m4 = scale2(m, 4.0f);
    const float2 tms = mul2(add2(sub2(m4.hi, s.hi), sub2(m4.lo, s.lo)), s.hi);
    dd2 r;
    r.hi.x = tms.x < 0.0f ? m4.hi.x : s.hi.x;
    r.lo.x = tms.x < 0.0f ? m4.lo.x : s.lo.x;
    r.hi.y = tms.y < 0.0f ? m4.hi.y : s.hi.y;
    r.lo.y = tms.y < 0.0f ? m4.lo.y : s.lo.y;
    r.hi.x = ab.x > 0.0f ? r.hi.x : 0.0f;
    r.lo.x = ab.x > 0.0f ? r.lo.x : 0.0f;
    r.hi.y = ab.y > 0.0f ? r.hi.y : 0.0f;
    r.lo.y = ab.y > 0.0f ? r.lo.y : 0.0f;
    return r;
}

// ---------------------------------------------------------------------------
// float64 -> double-float with integer operations, and back on the float64 pipe.
// ---------------------------------------------------------------------------
// x = hi + lo with hi = x rounded to 24 significand bits (half away from zero) and lo the rest
// rounded to float32 (|lo| <= 2^-25 |x|; the pair carries 48 of x's 53 bits, rounded to
// nearest).  |x| below 2^-74 (5.3e-23) is flushed to zero: populations here are O(1), so the
// absolute error stays below that.  Non-finite x and |x| >= 2^127 give +-inf or NaN in hi.
__device__ __forceinline__ dd dd_split(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hw = (unsigned)(b >> 32), lw = (unsigned)b;
    const unsigned ex = (hw >> 20) & 0x7FFu;
    const unsigned sign = hw & 0x80000000u;
    // top 24 significand bits with the exponent rebiased (1023 -> 127); a carry from the
    // rounding increment moves into the exponent field, as it should
    unsigned fb = (((hw & 0x7FFFFFFFu) - (896u << 20)) << 3) | (lw >> 29);
    const unsigned up = (lw >> 28) & 1u;
    fb += up;
    // remainder in units of 2^(ex - 1075): the low 29 bits, less 2^29 when hi was rounded up
    const int r = (int)(lw & 0x1FFFFFFFu) - (int)(up << 29);
    const float scale = __uint_as_float(((ex - 948u) & 0xFFu) << 23);   // 2^(ex - 1075) in range
    const float lo = __fmul_rn(__int2float_rn(r), scale);
    // selects, not branches: flushed, overflowing and non-finite inputs
    const bool tiny = ex < 949u, big = ex >= 1150u;
    const bool nan = ex == 2047u && ((hw & 0xFFFFFu) | lw) != 0u;
    const unsigned hbits = big ? (sign | 0x7F800000u | (nan ? 0x400000u : 0u)) : (fb | sign);
    return dd{tiny ? 0.0f : __uint_as_float(hbits),
              (tiny || big) ? 0.0f : __uint_as_float(__float_as_uint(lo) ^ sign)};
}

// dd_split of two values as a pair.  In the common range (2^-74 <= |x| < 2^127, tested once per
// pair) the rounding carry, the bias and the exponent field come from one 64-bit addition and a
// funnel shift: hi = the top 24 significand bits after adding half a unit, lo = the low 29 bits as
// a signed number (shifted left by 3, so that the conversion needs no sign extension) times the
// power of two of x's exponent.  The same values as dd_split, in 13 integer operations a value
// instead of about 28; everything else takes dd_split.
__device__ __forceinline__ dd2 dd_split2(double x, double y)
{
    const unsigned hx = (unsigned)__double2hiint(x), lx = (unsigned)__double2loint(x);
    const unsigned hy = (unsigned)__double2hiint(y), ly = (unsigned)__double2loint(y);
    auto top = [](unsigned h, unsigned l) {
        const unsigned long long t = (((unsigned long long)h << 32) | l) + 0xC800000010000000ull;   // - (896 << 52) + 2^28
        return __uint_as_float(((unsigned)(t >> 29) & 0x7FFFFFFFu) | (h & 0x80000000u));
    };
    auto pow2 = [](unsigned h) {   // +-2^(exponent of x)
        return __uint_as_float(((h * 8u + 0x40000000u) & 0x7F800000u) | (h & 0x80000000u));
    };
    dd2 r;
    r.hi = f2(top(hx, lx), top(hy, ly));
    const float2 rem = f2(__int2float_rn((int)(lx << 3)), __int2float_rn((int)(ly << 3)));
    r.lo = mul2(mul2(rem, f2(0x1p-55f, 0x1p-55f)), f2(pow2(hx), pow2(hy)));
    const bool okx = hx * 2u - (949u << 21) < (201u << 21), oky = hy * 2u - (949u << 21) < (201u << 21);
    if (!(okx && oky)) r = pack(dd_split(x), dd_split(y));
    return r;
}

// hi + lo rounded to float64 (to nearest, ties to even): both parts in float64 exactly, then one
// float64 addition rounds their sum.  hi is converted on the float64 pipe (1.9 lanes per cycle per
// SM; so infinities and NaN in hi carry over; next to an infinite hi a lo that is not finite reads as a
// finite number), lo by moving its fields with integer operations: three
// float64-pipe operations a value kept that pipe 55% busy over the step and more in the update,
// which waits for it (2048 x 2048: 0.588 ms, against 0.564 ms with two;
// rounding by integer additions instead took 0.591 ms for half of the values and 0.619 for all).
__device__ __forceinline__ double dd_to_double(dd v)
{
    const unsigned b = __float_as_uint(v.lo);
    const unsigned h = ((unsigned)((int)b >> 3) & 0x8FFFFFFFu) + 0x38000000u;
    return __dadd_rn((double)v.hi, __hiloint2double(v.lo == 0.0f ? 0 : (int)h, (int)(b << 29)));
}

}  // namespace lbm
