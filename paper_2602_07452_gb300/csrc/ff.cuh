// Paired-FP32 ("double-float") arithmetic for FP64-pipe-bound inner loops.
//
// A value is the unevaluated sum hi + lo of two floats with |lo| at most
// a few units in the last place of hi: some 48 significant bits.  Every
// operation is built from the error-free transformations of FP32 sums and
// products -- Knuth's TwoSum (TAOCP vol. 2, Sec. 4.2.2), Dekker's fast
// two-sum (1971) and the exact product error fmaf(a, b, -a b) -- so it runs on
// the FP32 pipe, which on this GPU issues 64 times the FP64 rate.  Sums use
// the short form (exact error of the high parts, plain sum of the low
// parts): a few units of 2^-48 relative when both operands have the same
// sign, and a few units of 2^-48 of |a| + |b| absolute in general.  Sums and
// products leave the pair unnormalized (no closing two-sum: |lo| stays within
// a few ulp of hi, which every operation here accepts, and the error of the
// short chains the deposit forms stays near 2^-45); the square root and the
// conversion from a double return normalized pairs.  The
// explicit __f*_rn intrinsics keep the compiler from contracting or
// reordering the transformations.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace fpic {

struct ff {
    float hi, lo;
};

// s + e of two floats with |a| >= |b| (or a == 0): exact.
__device__ __forceinline__ ff ff_fast2(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

// a + b of any two floats: exact.
__device__ __forceinline__ ff ff_sum2(float a, float b)
{
    const float s = __fadd_rn(a, b), v = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v))};
}

__device__ __forceinline__ ff ff_of(float a)
{
    return {a, 0.f};
}

// The double x as hi + lo, by integer operations on its bits (the FP64
// pipe's conversions would cost as much as FP64 arithmetic): hi is x rounded
// to a float -- sign, exponent (the biases differ by 896 = -128 modulo 256: the
// shifted field with its top bit flipped) and leading 23 fraction bits, one
// up when the remaining 29 bits reach a half -- and lo what that leaves, an
// integer of at most 2^28 rounded to a float, times 2^(e - 52): within 2^-50
// relative for 2^-98 <= |x| < 2^127; 0 below 2^-126 (and lo 0 below 2^-98),
// which only drops magnitudes far under the values this is used on.
constexpr unsigned F64_HI_2M126 = (1023u - 126u) << 20, F64_HI_2M98 = (1023u - 98u) << 20;

__device__ __forceinline__ ff ff_from(double x)
{
    const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
    const unsigned mag = hw & 0x7fffffffu;
    const unsigned h = ((__funnelshift_l(lw, hw, 3) ^ 0x40000000u) & 0x7fffffffu) | (hw & 0x80000000u);
    const float scale = __uint_as_float((h & 0xff800000u) - (28u << 23));       // +-2^(e - 28)
    const int m = (int)(lw << 3) >> 3;                                          // bits 0..28, signed
    const float lo = __fmul_rn(__fmul_rn(__int2float_rn(m), 5.9604644775390625e-8f), scale);
    if (mag < F64_HI_2M126) return {0.f, 0.f};
    if (mag < F64_HI_2M98) return {__uint_as_float(h), 0.f};
    return {__uint_as_float(h + ((lw >> 28) & 1u)), lo};
}

// The same with hi cut off instead of rounded (lo of its sign, up to an ulp of
// hi: the pair good to 2^-47): a few instructions fewer, for kernels bound by
// their issue slots; lo 0 below 2^-70.
__device__ __forceinline__ ff ff_cut(double x)
{
    const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
    const unsigned mag = hw & 0x7fffffffu;
    const unsigned h = ((__funnelshift_l(lw, hw, 3) ^ 0x40000000u) & 0x7fffffffu) | (hw & 0x80000000u);
    const float lo = __fmul_rn(__uint2float_rn(lw & 0x1fffffffu), __uint_as_float((h & 0xff800000u) - (52u << 23)));
    if (mag < F64_HI_2M126) return {0.f, 0.f};
    return {__uint_as_float(h), mag < ((1023u - 70u) << 20) ? 0.f : lo};
}

// A normal float (or 0) as a double, by integer operations on its bits.
__device__ __forceinline__ double f2d_bits(float f)
{
    const unsigned u = __float_as_uint(f);
    const unsigned e8 = (u >> 23) & 0xffu;
    if (e8 == 0u) return 0.0;
    const unsigned hw = (u & 0x80000000u) | ((e8 + 896u) << 20) | ((u & 0x7fffffu) >> 3);
    return __longlong_as_double((long long)(((unsigned long long)hw << 32) | ((unsigned long long)(u & 7u) << 29)));
}

__device__ __forceinline__ double ff_to(ff a)
{
    return f2d_bits(a.hi) + f2d_bits(a.lo);
}

// The pair's sum as a double by integer operations, off the FP64 pipe: h,
// the sum rounded towards zero, leaves a remainder of its own sign below one
// of its last places, which in units of the last place of h's double (2^(e -
// 52)) is an integer added to that double's bits; to 2^-47 relative.
__device__ __forceinline__ double ff_to_bits(ff a)
{
    const float h = __fadd_rz(a.hi, a.lo), l = __fadd_rn(__fsub_rn(a.hi, h), a.lo);
    const unsigned u = __float_as_uint(h), ex = u & 0x7f800000u;
    // l sign(h) 2^-e: the reciprocal power of two has the exponent field 254 - e8
    const float s = __uint_as_float((u & 0x80000000u) | ((254u << 23) - ex));
    const int off = __float2int_rn(__fmul_rn(__fmul_rn(l, s), 4503599627370496.f));
    const unsigned hw = (u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20));
    const long long b = (long long)(((unsigned long long)hw << 32) | (u << 29)) + off;
    return ex ? __longlong_as_double(b) : 0.0;
}

__device__ __forceinline__ ff ff_add(ff a, ff b)
{
    const float s = __fadd_rn(a.hi, b.hi);
    const float v = __fsub_rn(s, a.hi);
    const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, v)), __fsub_rn(b.hi, v));
    return {s, __fadd_rn(e, __fadd_rn(a.lo, b.lo))};
}

// a + b when a_hi >= b_hi >= 0 (more generally: a_hi's exponent at least
// b_hi's): Dekker's fast two-sum of the high parts gives the same sum and
// the same exact error as the two-sum in ff_add, so the same pair, with
// three additions fewer.
__device__ __forceinline__ ff ff_add_ge(ff a, ff b)
{
    const float s = __fadd_rn(a.hi, b.hi);
    return {s, __fadd_rn(__fsub_rn(b.hi, __fsub_rn(s, a.hi)), __fadd_rn(a.lo, b.lo))};
}

__device__ __forceinline__ ff ff_neg(ff a)
{
    return {-a.hi, -a.lo};
}

__device__ __forceinline__ ff ff_mul(ff a, ff b)
{
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    return {p, __fmaf_rn(a.lo, b.hi, e)};
}

__device__ __forceinline__ ff ff_sqr(ff a)
{
    const float p = __fmul_rn(a.hi, a.hi);
    const float e = __fmaf_rn(a.hi, a.hi, -p);
    return {p, __fmaf_rn(__fadd_rn(a.hi, a.hi), a.lo, e)};
}

// a times a float b
__device__ __forceinline__ ff ff_mulf(ff a, float b)
{
    const float p = __fmul_rn(a.hi, b);
    return {p, __fmaf_rn(a.lo, b, __fmaf_rn(a.hi, b, -p))};
}

// a times a power of two (exact)
__device__ __forceinline__ ff ff_scale(ff a, float two_k)
{
    return {__fmul_rn(a.hi, two_k), __fmul_rn(a.lo, two_k)};
}

// sqrt(a) for a > 0 in the normal float range.  With the FP32 estimate y
// of 1/sqrt(a_hi) (relative error e up to 2 ulp, about 2^-22), s = a_hi y
// is corrected by one Newton step for the square root, s + (a - s^2) y / 2,
// with a - s^2 formed exactly from the product error of s^2 (a_hi - s^2 is
// exact: the two are within a factor 2).  The step leaves 3 e^2 / 2 of the
// estimate's error (at most about 2^-43.4) beside the roundings of the
// correction (about 2^-46): ample for the deposit's lattices, whose
// shares are held to 1e-10 (fpic_probe_math measures it).
__device__ __forceinline__ ff ff_sqrt(ff a)
{
    const float y = rsqrtf(a.hi);
    const float s = __fmul_rn(a.hi, y);
    const float p = __fmul_rn(s, s);
    const float pe = __fmaf_rn(s, s, -p);
    const float d = __fadd_rn(__fsub_rn(__fsub_rn(a.hi, p), pe), a.lo);
    return ff_fast2(s, __fmul_rn(d, __fmul_rn(0.5f, y)));
}

// 1/a for a > 0 in the normal float range: the FP32 estimate y of 1/a_hi
// (relative error about 2^-23), once corrected in FP32 (y (1 + e), e = 1 - a_hi
// y by a fused multiply-add: half an ulp), then e = 1 - a y from the exact
// product error of a_hi y (1 - a_hi y is exact: the two are within a factor
// 2 of 1), and 1/a = y / (1 - e) = y (1 + e + e^2 + ...) to second order:
// relative error about 2^-47 (the roundings of e and y (e + e^2));
// fpic_probe_math measures it.
__device__ __forceinline__ ff ff_rcp(ff a)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a.hi));
    y = __fmaf_rn(y, __fmaf_rn(-a.hi, y, 1.f), y);
    const float p = __fmul_rn(a.hi, y);
    const float e = __fsub_rn(__fsub_rn(__fsub_rn(1.f, p), __fmaf_rn(a.hi, y, -p)), __fmul_rn(a.lo, y));
    return ff_fast2(y, __fmul_rn(y, __fmaf_rn(e, e, e)));
}

}  // namespace fpic
