// Floating-point numbers of some 60 significant bits in integer registers: a
// value is m 2^e with a 64-bit signed m, |m| < 2^62, normalised when |m| >=
// 2^61.  The right-hand side of the equations of motion runs on these
// because the FP64 pipe takes 64 issue slots per instruction, while a product
// here is about ten integer instructions and a sum about eleven (measured 23
// and 8 to 15 slots a warp; the same in three floats 30 and 26, an FP64
// fused multiply-add 63), and it carries ten bits more than a double, so
// that results rounded once to a double are closer to the exact ones than a
// chain of FP64 operations.  Products and sums drop at most one leading bit
// each (and what a sum cancels) and are not normalised again; x_norm restores
// them.  No infinities or NaNs: callers keep those to the FP64 forms.
#pragma once

#include <stdint.h>
#include <string.h>

namespace fpic {

#define FPIC_HD __host__ __device__ __forceinline__

struct xf {
    long long m;
    int e;
};

constexpr int XF_ZERO_E = -200000;     // exponent of a zero: below every product of a few values

FPIC_HD int x_hi(long long m)
{
    return (int)(m >> 32);
}

FPIC_HD int x_mulhi(int a, int b)
{
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return (int)(((long long)a * b) >> 32);
#endif
}

FPIC_HD unsigned x_umulhi(unsigned a, unsigned b)
{
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (unsigned)(((unsigned long long)a * b) >> 32);
#endif
}

FPIC_HD int x_clz(unsigned v)
{
#ifdef __CUDA_ARCH__
    return __clz((int)v);
#else
    return v ? __builtin_clz(v) : 32;
#endif
}

FPIC_HD unsigned long long x_bits(double d)
{
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(d);
#else
    unsigned long long u;
    memcpy(&u, &d, 8);
    return u;
#endif
}

FPIC_HD double x_double(unsigned long long u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double d;
    memcpy(&d, &u, 8);
    return d;
#endif
}

// A finite double; zeros and subnormals become an m with an exponent below
// everything.  Negative values as the complement (off by 2^-61 of the value).
FPIC_HD xf x_from(double d)
{
    const unsigned long long b = x_bits(d);
    const unsigned hw = (unsigned)(b >> 32), lw = (unsigned)b;
    const unsigned s = (unsigned)((int)hw >> 31), E = (hw >> 20) & 0x7ffu;
    const unsigned h = ((((hw & 0xfffffu) | 0x100000u) << 9) | (lw >> 23)) ^ s, l = (lw << 9) ^ s;
    return {(long long)(((unsigned long long)h << 32) | l), E ? (int)E - 1084 : XF_ZERO_E};
}

// the same for a positive normal d
FPIC_HD xf x_from_pos(double d)
{
    const unsigned long long b = x_bits(d);
    const unsigned hw = (unsigned)(b >> 32), lw = (unsigned)b;
    const unsigned h = (((hw & 0xfffffu) | 0x100000u) << 9) | (lw >> 23);
    return {(long long)(((unsigned long long)h << 32) | (lw << 9)), (int)(hw >> 20) - 1084};
}

// Rounded to the nearest double; 0 below the normal range, infinite above it.
// Out of line: a right-hand side converts six of them, and its code is long
// for the instruction cache (2 to 3 % of a push).
static __host__ __device__ __noinline__ double x_to(xf a)
{
    const unsigned long long s = (unsigned long long)(a.m >> 63);
    unsigned long long u = (unsigned long long)a.m ^ s;
    int e = a.e;
    if ((u >> 32) == 0) {              // cancelled to the low word
        u <<= 32;
        e -= 32;
    }
    const int n = x_clz((unsigned)(u >> 32));
    if (n == 32) return 0.0;
    u <<= n;
    const int E = 1085 + e - n;        // biased exponent less one: the leading bit adds one
    const unsigned long long r = (u >> 11) + ((u >> 10) & 1u);
    if ((unsigned)E >= 2046u) return E < 0 ? 0.0 : x_double((s & 0x8000000000000000ull) | 0x7ff0000000000000ull);
    return x_double((s & 0x8000000000000000ull) | (r + ((unsigned long long)(unsigned)E << 52)));
}

FPIC_HD xf x_norm(xf a)
{
    const int h = x_hi(a.m), n = x_clz((unsigned)(h ^ (h >> 31))) - 2;
    return {(long long)((unsigned long long)a.m << n), a.e - n};
}

// a b + c / 2^32 of signed integers
FPIC_HD int x_madhi(int a, int b, int c)
{
#ifdef __CUDA_ARCH__
    int d;
    asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
#else
    return x_mulhi(a, b) + c;
#endif
}

// m1 m2 / 2^62: the high words of 2 m1 and 2 m2 times each other, and the
// cross terms with half their low words (which stay signed); to a few units of m.
FPIC_HD int x_h2(long long m)
{
    return x_hi((long long)((unsigned long long)m << 1));
}

FPIC_HD int x_l2(long long m)
{
    return (int)((unsigned)m & 0x7fffffffu);
}

FPIC_HD xf x_mul(xf a, xf b)
{
    const int ha = x_h2(a.m), hb = x_h2(b.m);
    const long long c = x_madhi(ha, x_l2(b.m), x_mulhi(hb, x_l2(a.m)));
    return {(long long)ha * hb + 2 * c, a.e + b.e + 62};
}

FPIC_HD xf x_sqr(xf a)
{
    const int ha = x_h2(a.m);
    const long long c = x_mulhi(ha, x_l2(a.m));
    return {(long long)ha * ha + 4 * c, 2 * a.e + 62};
}

FPIC_HD xf x_neg(xf a)
{
    return {~a.m, a.e};
}

// m >> n, the sign for n above 63
FPIC_HD long long x_shr(long long m, int n)
{
#ifdef __CUDA_ARCH__
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(n));
    return r;
#else
    return m >> (n < 63 ? n : 63);
#endif
}

FPIC_HD xf x_add(xf a, xf b)
{
    const int e = (a.e > b.e ? a.e : b.e) + 1;
    return {x_shr(a.m, e - a.e) + x_shr(b.m, e - b.e), e};
}

// a + b + c in one alignment (two leading bits dropped at most)
FPIC_HD xf x_add3(xf a, xf b, xf c)
{
    const int ab = a.e > b.e ? a.e : b.e, e = (ab > c.e ? ab : c.e) + 2;
    return {x_shr(a.m, e - a.e) + x_shr(b.m, e - b.e) + x_shr(c.m, e - c.e), e};
}

FPIC_HD xf x_pow2(int k)              // 2^k
{
    return {0x2000000000000000ll, k - 61};
}

// E Y / 2^32 of a 64-bit E and Y in [0, 2^31)
FPIC_HD long long x_scale32(long long E, unsigned Y)
{
    return (long long)x_hi(E) * (int)Y + (long long)x_umulhi((unsigned)E, Y);
}

FPIC_HD float x_float(unsigned u)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float f;
    memcpy(&f, &u, 4);
    return f;
#endif
}

FPIC_HD unsigned x_float_bits(float f)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(f);
#else
    unsigned u;
    memcpy(&u, &f, 4);
    return u;
#endif
}

// The FP32 estimate in units of 2^-24, for a value of at least 1/2 and below 1.  The
// hardware's may fall an ulp or two outside (its documented error is an ulp for
// the reciprocal and 2^-22.9 for the root): below 1/2, where an ulp is half a
// unit, counting down in whole ones is as good an estimate; at 1 it is held
// below.
FPIC_HD unsigned x_est24(float y)
{
    const unsigned u = x_float_bits(y);
    return (u < 0x3f7fffffu ? u : 0x3f7fffffu) - 0x3e800000u;
}

// 1/a for a > 0: with X = m / 2^61 in [1, 2), the FP32 estimate Y of 1/X in 31
// fraction bits, e = 1 - X Y exact to 2^-61 and Y (1 + e + e^2): e is below
// 2^-21, the next term below 2^-63.  a normalised, y the estimate of 1 / x_rcp_arg(a).
FPIC_HD float x_rcp_arg(xf a)
{
    return x_float(0x3f800000u | (((unsigned)x_hi((long long)((unsigned long long)a.m << 1)) >> 7) & 0x7fffffu));
}

FPIC_HD xf x_rcp_est(xf a, float y)
{
    const unsigned long long m = (unsigned long long)a.m << 1;
    const int h = x_hi((long long)m);
    const unsigned Y = x_est24(y) << 7;
    const long long p = (long long)h * (int)Y + (long long)x_umulhi((unsigned)m, Y);
    const long long E = 0x2000000000000000ll - p;                       // e 2^61
    const int e12 = (int)(E >> 12), t = x_mulhi(e12, e12);              // e 2^49, e^2 2^66
    const int t2 = x_mulhi(t << 6, (int)Y) >> 11;                       // Y e^2 2^60
    const long long r = ((long long)Y << 29) + (x_scale32(E, Y) + t2);  // 2^60 / X
    return {r << 1, -122 - a.e};
}

FPIC_HD xf x_rcp(xf a)
{
    a = x_norm(a);
    const float x = x_rcp_arg(a);
    float y;
#ifdef __CUDA_ARCH__
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
#else
    y = 1.f / x;
#endif
    return x_rcp_est(a, y);
}

// 1/sqrt(a) for a > 0 in the same way: X in [1, 4) (an even exponent), e = 1 -
// X Y^2 with Y of 24 bits (Y^2 exact), Y (1 + e/2 + 3 e^2/8).
FPIC_HD float x_rsqrt_arg(xf a)
{
    const unsigned odd = (unsigned)(a.e + 61) & 1u;
    return x_float(x_float_bits(x_rcp_arg(a)) + (odd << 23));
}

FPIC_HD xf x_rsqrt_est(xf a, float y)
{
    const unsigned long long m = (unsigned long long)a.m << 1;
    const int h = x_hi((long long)m), E0 = a.e + 61, odd = E0 & 1;
    const unsigned y24 = x_est24(y), Y = y24 << 7;
    const long long y2 = (long long)((unsigned long long)y24 * y24 << 14);   // Y^2 2^62
    const int hy = x_hi(y2), ly = (int)((unsigned)y2 >> 1), la = (int)((unsigned)m >> 1);
    const long long c = x_mulhi(h, ly) + x_mulhi(hy, la);
    const long long p = (long long)h * hy + 2 * c;                           // (m / 2^62) Y^2 2^60
    const long long E = 0x1000000000000000ll - (p << odd);                   // e 2^60
    const int e11 = (int)(E >> 11), t = x_mulhi(e11, e11);                   // e 2^49, e^2 2^66
    const int t2 = x_mulhi((3 * t) << 4, (int)Y) >> 12;                      // 3/8 Y e^2 2^60
    const long long r = ((long long)Y << 29) + (x_scale32(E, Y) + t2);
    return {r << 1, -61 - (E0 >> 1)};
}

FPIC_HD xf x_rsqrt(xf a)
{
    a = x_norm(a);
    const float x = x_rsqrt_arg(a);
    float y;
#ifdef __CUDA_ARCH__
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
#else
    y = (float)(1.0 / __builtin_sqrt((double)x));
#endif
    return x_rsqrt_est(a, y);
}

}  // namespace fpic
