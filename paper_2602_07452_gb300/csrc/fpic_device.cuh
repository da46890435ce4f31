// Device-side building blocks of the GRPIC push: closed-form Kerr-Schild
// metric and derivatives (Appendix A), the equations of motion (Eqs. p1, p2,
// O1, O2), the Hamiltonian (Eq. Ham) and the staggered-grid field gather.
//
// GB300 note: FP64 issues at 1/64 of the FP32 rate, so the right-hand side
// runs on integer mantissas of 60 bits (rhs_x, xf.cuh; the FP64 form remains
// for arguments that have none), the sin/cos series of small steps and the
// corrections of reciprocals and roots in paired FP32 (ff.cuh), and cell
// location by integer comparison of the IEEE bit patterns (order-preserving)
// instead of FP64 compares.  The field gather and the stages' sums are FP64,
// fused multiply-adds throughout.  Against an extended-precision RK4 step the
// pushed states' relative errors are 4.8e-17 to 5.1e-17 at 48 to 900 cells a
// side, H's 7e-17 to 9e-17 (all in FP64 16e-17).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "ff.cuh"
#include "xf.cuh"

namespace fpic {

struct BH {
    double M, a, a2, twoM;
};

// 1/x and 1/sqrt(x) with two FP64-pipe operations each.  The FP32 estimate y
// of the result is a double with 24 significant bits, so that the residual
// e = 1 - x y (e = 1 - x y^2, y^2 exact in 48 bits) is one fused multiply-add,
// good to 2^-53 of itself; the correction y (e + e^2) (y (e/2 + 3 e^2/8)) of
// the binomial series -- e is about 2^-21, the next term below 2^-64 -- needs
// 32 significant bits and is formed in paired FP32, and one FP64 addition
// rounds the result: within an ulp (fpic_probe_math measures both).  The
// FP64 pipe takes 64 issue slots per operation, so the 40 or so FP32 and
// integer instructions cost less than the two (three) FP64 operations they
// replace.  Arguments outside 2^-60 .. 2^60 (where the correction's low float
// keeps its bits), zeros, infinities and NaNs take the FP64 forms: the hardware
// estimate y and y (1 + e + e^2), or y (1 + e/2 + 3 e^2/8).
__device__ __forceinline__ bool f32_range(unsigned hi)      // 2^-60 <= x < 2^60, hi the high word of |x|
{
    return hi - ((1023u - 60u) << 20) < (120u << 20);
}

// a double in the float range as a float, cut off; a normal float as a double
__device__ __forceinline__ float f32_cut(double x)
{
    const unsigned hw = (unsigned)__double2hiint(x);
    return __uint_as_float(((__funnelshift_l((unsigned)__double2loint(x), hw, 3) ^ 0x40000000u) & 0x7fffffffu) |
                           (hw & 0x80000000u));
}

__device__ __forceinline__ double f64_of(float y)
{
    const unsigned u = __float_as_uint(y);
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}

static __device__ __noinline__ double rcp_wide(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

static __device__ __noinline__ double rsqrt_wide(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x * y, y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);
}

__device__ __forceinline__ double rcp_nr(double x)
{
    if (!f32_range((unsigned)__double2hiint(x) & 0x7fffffffu)) return rcp_wide(x);
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f32_cut(x)));
    const double yd = f64_of(y);
    const ff e = ff_from(fma(-x, yd, 1.0));
    return yd + ff_to_bits(ff_mulf({e.hi, __fmaf_rn(e.hi, e.hi, e.lo)}, y));
}

__device__ __forceinline__ double rsqrt_nr(double x)
{
    if (!f32_range((unsigned)__double2hiint(x))) return rsqrt_wide(x);       // negative x too
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f32_cut(x)));
    // y^2 = m^2 2^(2 E - 46), m in [2^23, 2^24): its leading bit is bit 46 + k of m^2
    const unsigned u = __float_as_uint(y), m = (u & 0x7fffffu) | 0x800000u;
    const unsigned long long M = (unsigned long long)m * m;
    const unsigned k = (unsigned)(M >> 47);
    const unsigned long long b = (M << (6 - k)) + ((unsigned long long)((2u * (u >> 23) + 768u + k) << 20) << 32);
    const ff e = ff_from(fma(-x, __longlong_as_double((long long)b), 1.0));
    const ff c = ff_mulf({0.5f * e.hi, __fmaf_rn(0.375f * e.hi, e.hi, 0.5f * e.lo)}, y);
    return f64_of(y) + ff_to_bits(c);
}

// Square root of a positive normal x (the deposit's trapezoid sums): the
// hardware reciprocal-square-root estimate y refined by one coupled Newton
// step on (g, h) = (x y, y / 2) (Goldschmidt's iteration, e.g. Markstein,
// IA-64 and Elementary Functions, 2000): g (1 + r), r = 1/2 - g h, squares
// the estimate's relative error; fpic_probe_math measures at most 1.3e-12
// (2^-39.6) against correctly rounded square roots, far inside the deposit's
// 1e-10 bound.  Each particle's shares still sum to its charge to rounding:
// they are ratios of the same subvolumes.
// sqrt2_dep returns 2 sqrt(x) in the same step written as g (3 - g y) with
// g = x y: three FP64 operations after the estimate; the deposit only uses
// ratios of sums of these values, so the factor 2 cancels.
__device__ __forceinline__ double sqrt2_dep(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double g = x * y;
    return g * fma(-g, y, 3.0);
}

__device__ __forceinline__ double sqrt_dep(double x)
{
    return 0.5 * sqrt2_dep(x);
}

// sin h and cos h - 1 for a step h inside one cell: Maclaurin series through
// h^5 / h^6 when |h| < 2^-10 (the first omitted terms are below 2^-62 of
// sin h and 2^-63 of cos h - 1), through h^7 / h^8 when |h| < 2^-7 (below
// 1e-22 relative), else libm.
// |x| < 2^e for a power of two 2^e whose double has high word hi_pow2 (and
// low word 0): the same result as the FP64 compare (false for a NaN), from
// the high word by one integer compare, off the FP64 pipe.
__device__ __forceinline__ bool abs_below_pow2(double x, unsigned hi_pow2)
{
    return ((unsigned)__double2hiint(x) & 0x7fffffffu) < hi_pow2;
}
constexpr unsigned HI_2M10 = 0x3f500000u, HI_2M7 = 0x3f800000u;   // 2^-10, 2^-7

__device__ __forceinline__ void sincos_step(double h, double& sh, double& cm)
{
    if (abs_below_pow2(h, HI_2M10)) {
        const double h2 = h * h;
        sh = h * fma(h2, fma(h2, 1.0 / 120.0, -1.0 / 6.0), 1.0);
        cm = h2 * fma(h2, fma(h2, -1.0 / 720.0, 1.0 / 24.0), -0.5);
    } else if (abs_below_pow2(h, HI_2M7)) {
        const double h2 = h * h;
        sh = h * fma(h2, fma(h2, fma(h2, -1.0 / 5040.0, 1.0 / 120.0), -1.0 / 6.0), 1.0);
        cm = h2 * fma(h2, fma(h2, fma(h2, 1.0 / 40320.0, -1.0 / 720.0), 1.0 / 24.0), -0.5);
    } else {
        double s, c;
        sincos(h, &s, &c);
        sh = s;
        cm = c - 1.0;
    }
}

// sin h and cos h - 1 of a step h in paired FP32 (the deposit's th
// lattice rotations).  Below 2^-7 by the Maclaurin series: h - h^3/6 and
// -h^2/2 in paired arithmetic, the next terms (h^5/120; h^4/24 - h^6/720),
// below 2^-28 relative, in FP32, the omitted ones below 2^-48 of the
// result: sin h to about 2^-46 relative, cos h - 1 to about 2^-40 of
// itself (2^-55 absolute, which is what the rotations need); larger steps
// (coarse grids) through the FP64 routine sincos_step.
__device__ __forceinline__ void sincos_step_ff(ff h, ff& sh, ff& cm)
{
    if (fabsf(h.hi) >= 0.0078125f) {
        double s, c;
        sincos_step(ff_to(h), s, c);
        sh = ff_from(s);
        cm = ff_from(c);
        return;
    }
    const ff t = ff_sqr(h);
    const ff h3 = ff_mul(h, t);
    const ff sixth = {__uint_as_float(0x3e2aaaabu), __uint_as_float(0xb1aaaaabu)};   // 1/6
    const float h5 = __fmul_rn(__fmul_rn(h3.hi, t.hi), 1.f / 120.f);
    sh = ff_add(h, ff_add(ff_neg(ff_mul(h3, sixth)), ff_of(h5)));
    const float c4 = __fmul_rn(__fmul_rn(t.hi, t.hi), __fsub_rn(1.f / 24.f, __fmul_rn(t.hi, 1.f / 720.f)));
    cm = ff_add(ff_scale(t, -0.5f), ff_of(c4));
}

__device__ __forceinline__ void sincos_step_ff(double hd, ff& sh, ff& cm)
{
    sincos_step_ff(ff_from(hd), sh, cm);
}

static __device__ __noinline__ double2 sincos_far(double t)
{
    double2 v;
    sincos(t, &v.x, &v.y);
    return v;
}

// sin and cos of t from those of a nearby t0 by the angle-addition formula,
// with sin d and cos d - 1 of d = t - t0 by their Taylor series (the first
// omitted terms are below 1e-23 for |d| < 2^-7); farther away, sincos.  The
// series run in paired FP32: cos d - 1 and sin d - d are below 2^-15 and 2^-23,
// so their 46 bits leave errors under 2^-60 and 2^-68 of the result; FP64 does
// the difference, d + (sin d - d) and the rotation: six operations.
__device__ __forceinline__ void sincos_near(double t0, double s0, double c0, double t, double& s, double& c)
{
    const double d = t - t0;
    if (abs_below_pow2(d, HI_2M7)) {
        const ff f = ff_from(d), q = ff_sqr(f);
        const ff sixth = {__uint_as_float(0x3e2aaaabu), __uint_as_float(0xb1aaaaabu)};   // 1/6
        // sin d - d = -d^3/6 (1 - d^2/20 + d^4/840), cos d - 1 = -d^2/2 + d^4/24 - d^6/720 + d^8/40320
        ff b = ff_neg(ff_mul(ff_mul(f, q), sixth));
        b.lo = __fmaf_rn(__fmul_rn(b.hi, q.hi), __fmaf_rn(q.hi, 1.f / 840.f, -0.05f), b.lo);
        const float q2 = __fmul_rn(q.hi, q.hi);
        const ff m = {-0.5f * q.hi, __fmaf_rn(q2, __fmaf_rn(q.hi, __fmaf_rn(q.hi, 1.f / 40320.f, -1.f / 720.f), 1.f / 24.f),
                                              -0.5f * q.lo)};
        const double sd = d + ff_to_bits(b), cm = ff_to_bits(m);
        s = fma(s0, cm, fma(c0, sd, s0));
        c = fma(c0, cm, fma(-s0, sd, c0));
    } else {
        const double2 v = sincos_far(t);
        s = v.x;
        c = v.y;
    }
}

// Metric at a point (r, th) given sin/cos th.
struct Geo {
    double s, c, s2, c2, r2, rho2, irho2, t;  // t = 1/(rho^2 sin^2 th)
    double twoMr, a2s2;               // 2 M r, a^2 sin^2 th
    double xi, alpha, ixi, beta;
    double gurr, gurp, gutt, gupp;
    double grr, grp, gtt, gpp, sqrtg;
};

// With xi = 1 + 2 M r / rho^2: alpha = xi^(-1/2), beta^r = 2 M r / (rho^2 xi)
// = 1 - 1/xi, g^rr = a^2 s^2 / rho^2 + 1/xi, g^rp = a / rho^2,
// g^tt = 1 / rho^2, g^pp = 1 / (rho^2 s^2) (App. A).
__device__ __forceinline__ void geo_eval(const BH& bh, double r, double s, double c, Geo& g)
{
    const double s2 = s * s, c2 = c * c;
    g.s = s;
    g.c = c;
    g.s2 = s2;
    g.c2 = c2;
    g.r2 = r * r;
    g.rho2 = fma(bh.a2, c2, g.r2);
    g.t = rcp_nr(g.rho2 * s2);
    g.irho2 = g.t * s2;
    g.twoMr = bh.twoM * r;
    g.a2s2 = bh.a2 * s2;
    g.xi = fma(g.twoMr, g.irho2, 1.0);
    g.alpha = rsqrt_nr(g.xi);
    g.ixi = g.alpha * g.alpha;
    g.beta = 1.0 - g.ixi;
    g.gurr = fma(g.a2s2, g.irho2, g.ixi);
    g.gurp = bh.a * g.irho2;
    g.gutt = g.irho2;
    g.gupp = g.t;
    g.grr = g.xi;
    g.grp = -bh.a * g.xi * s2;
    g.gtt = g.rho2;
    g.gpp = s2 * fma(bh.a2 * g.xi, s2, g.rho2);
    g.sqrtg = g.rho2 * g.xi * g.alpha * s;
}

// FP32 value of a double from its high word (20 of its 52 mantissa bits,
// truncated), by integer operations only, for the index estimates of
// locate: no FP64 conversion instruction.  Exact enough for normal floats;
// any other input still ends in the right cell, since the walk in locate
// corrects any start.
__device__ __forceinline__ float f32_est(double x)
{
    const int hi = __double2hiint(x);
    const int e = ((hi >> 20) & 0x7ff) - 896;
    return __int_as_float((hi & (int)0x80000000) | (e << 23) | ((hi & 0xfffff) << 3));
}

// For a, b >= 0 or NaN (update sizes, tolerances): a <= b and a < b as the
// FP64 compares give them (false when either is a NaN), and fmax(m, a) for a
// running maximum m >= 0 (a NaN a is ignored), by integer compares of the
// bit patterns -- non-negative doubles order like their bits -- off the
// FP64 pipe.
constexpr long long F64_INF_BITS = 0x7ff0000000000000LL;
__device__ __forceinline__ bool le_nonneg(double a, double b)
{
    const long long ba = __double_as_longlong(a), bb = __double_as_longlong(b);
    return ba <= bb && bb <= F64_INF_BITS;
}
__device__ __forceinline__ bool lt_nonneg(double a, double b)
{
    const long long ba = __double_as_longlong(a), bb = __double_as_longlong(b);
    return ba < bb && bb <= F64_INF_BITS;
}
__device__ __forceinline__ double fmax_nonneg(double m, double a)
{
    const long long bm = __double_as_longlong(m), ba = __double_as_longlong(a);
    return (ba > F64_INF_BITS || ba <= bm) ? m : a;
}

// x != 0 and x < 0 as the FP64 compares give them, by integer compares.
__device__ __forceinline__ bool not_zero(double x)
{
    return ((unsigned long long)__double_as_longlong(x) << 1) != 0ull;
}
__device__ __forceinline__ bool is_neg(double x)
{
    const unsigned long long m = (unsigned long long)__double_as_longlong(x) << 1;
    return __double_as_longlong(x) < 0 && m - 1ull < 0xffe0000000000000ull;
}

// x / 2 by taking one from the exponent, off the FP64 pipe; zeros, numbers
// near or below the normal range, infinities and NaNs go through the
// multiplication: the product's value for every x.
__device__ __forceinline__ double half_of(double x)
{
    const unsigned e = (unsigned)__double2hiint(x) & 0x7ff00000u;
    if (e - 0x00200000u < 0x7fd00000u) return __hiloint2double(__double2hiint(x) - 0x00100000, __double2loint(x));
    return 0.5 * x;
}

// x == 1 by an integer compare.
__device__ __forceinline__ bool is_one(double x)
{
    return __double_as_longlong(x) == 0x3ff0000000000000LL;
}

// Order-preserving integer key of a double (monotone for all non-NaN values).
__device__ __forceinline__ long long okey(double x)
{
    long long b = __double_as_longlong(x);
    return b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
}

// Grid as seen by the kernels.  Node tables and their inverse spacings
// 1/(X[i+1]-X[i]) live in library-owned device memory.
struct GridDev {
    int Nr, Nth, ld;
    const double *rn, *rh, *tn, *th;   // th: Nth half nodes + th[Nth] = th[0] + (tn[Nth] - tn[0])
    const double *irn, *irh, *itn, *ith;
    float lr0, lrh0, ilr;        // FP32 index estimate in ln r
    float t0, th0, it;           // FP32 index estimate in th
    int full;                    // full-theta domain (periodic th), else half-theta
    double tlo, tper, thlo;      // tn[0], the period tn[Nth] - tn[0], th[0]
};

// The th a gather sees.  Half-theta domain: th itself on both sub-grids,
// Nth half nodes.  Full-theta domain (Sec. 2.5: periodic boundaries): th
// wrapped into [tn[0], tn[0] + P) on the node sub-grid; on the half-node
// sub-grid a point below th[0] is taken at th + P, in the wrap cell
// [th[Nth-1], th[Nth] = th[0] + P] whose upper column (Nth) holds the image
// of column 0, so that sub-grid has Nth + 1 nodes.  One wrap suffices:
// particle states stay in the period and the RK4 stages and IMR midpoints
// stay within a step of it.
// The full-theta wrap is kept out of line behind a warp-uniform branch: if
// it were if-converted, its FP64 compares and adds would be issued in the
// half-theta domain too, on an FP64-bound push.
static __device__ __noinline__ double2 theta_wrap_full(double th, double tlo, double tper, double thlo)
{
    double t = th < tlo ? th + tper : th;
    t = t >= tlo + tper ? t - tper : t;
    return make_double2(t, t < thlo ? t + tper : t);
}

__device__ __forceinline__ void theta_views(const GridDev& G, double th, double& tn_view, double& th_view, int& mh)
{
    if (G.full) {
        const double2 v = theta_wrap_full(th, G.tlo, G.tper, G.thlo);
        tn_view = v.x;
        th_view = v.y;
        mh = G.Nth + 1;
    } else {
        tn_view = th_view = th;
        mh = G.Nth;
    }
}

// Locate x in node list X[0..m-1]: X[i] <= x < X[i+1], clamped to
// [0, m-2]; w is the clamped linear weight.  est: FP32 index estimate.
__device__ __forceinline__ int locate_walk(const double* __restrict__ X, int m, long long kx, float est)
{
    int k = __float2int_rd(est);
    k = max(0, min(k, m - 2));
    // walk to the right cell (the estimate is within one cell on uniform grids)
    for (int it = 0; it < m && k > 0 && kx < okey(__ldg(X + k)); ++it) --k;
    for (int it = 0; it < m && k < m - 2 && kx >= okey(__ldg(X + k + 1)); ++it) ++k;
    return k;
}

__device__ __forceinline__ void locate(const double* __restrict__ X, const double* __restrict__ iX,
                                       int m, double x, float est, int& i, double& w)
{
    const long long kx = okey(x);
    const int k = locate_walk(X, m, kx, est);
    i = k;
    const double x0 = __ldg(X + k);
    double ww = (x - x0) * __ldg(iX + k);
    const bool below = kx < okey(x0);
    const bool above = kx >= okey(__ldg(X + k + 1));
    ww = below ? 0.0 : ww;
    ww = above ? 1.0 : ww;
    w = ww;
}

// The same without walking, for the gather: the weight is a NaN (an integer
// compare away) where the estimated cell is not x's, once in some ten thousand
// on grids even in ln r and th.  (Walks in the push's main path took a twentieth
// of its time, and a flag as much.)
__device__ __forceinline__ void locate_est(const double* __restrict__ X, const double* __restrict__ iX, int m, double x,
                                           float est, int& i, double& w)
{
    const long long kx = okey(x);
    const int k = max(0, min(__float2int_rd(est), m - 2));
    const double x0 = __ldg(X + k), x1 = __ldg(X + k + 1);
    const double wrong = __longlong_as_double(0x7fffffffffffffffLL);
    i = k;
    w = (x - x0) * __ldg(iX + k);
    if (kx < okey(x0)) w = k > 0 ? wrong : 0.0;
    if (kx >= okey(x1)) w = k < m - 2 ? wrong : 1.0;
}

__device__ __forceinline__ bool is_nan(double x)
{
    return (unsigned long long)(__double_as_longlong(x) << 1) > 0xffe0000000000000ull;
}

struct Fields {
    const double* f[6];   // D^r, D^th, D^ph, B^r, B^th, B^ph (Yee layout)
};

// Bilinear (r, th) gather of the six components at (r, th), all in FP64.
static __device__ __noinline__ void gather(const GridDev& G, const Fields& F, double r, double th, double v[6])
{
    const float lr = __logf(f32_est(r));
    int i0, i1, j0, j1;
    double wr0, wr1, wt0, wt1;
    locate(G.rn, G.irn, G.Nr + 1, r, (lr - G.lr0) * G.ilr, i0, wr0);
    locate(G.rh, G.irh, G.Nr, r, (lr - G.lrh0) * G.ilr, i1, wr1);
    double tnv, thv;
    int mh;
    theta_views(G, th, tnv, thv, mh);
    const float tfn = f32_est(tnv), tfh = G.full ? f32_est(thv) : tfn;
    locate(G.tn, G.itn, G.Nth + 1, tnv, (tfn - G.t0) * G.it, j0, wt0);
    locate(G.th, G.ith, mh, thv, (tfh - G.th0) * G.it, j1, wt1);
    const int ld = G.ld;
    // component k sits at (roff, toff): D^r (1,0) D^th (0,1) D^ph (0,0)
    //                                    B^r (0,1) B^th (1,0) B^ph (1,1)
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const bool ro = (k == 0 || k == 4 || k == 5);
        const bool to = (k == 1 || k == 3 || k == 5);
        const int i = ro ? i1 : i0, j = to ? j1 : j0;
        const double wr = ro ? wr1 : wr0, wt = to ? wt1 : wt0;
        const double* p = F.f[k] + (size_t)i * ld + j;
        const double f00 = __ldg(p), f01 = __ldg(p + 1);
        const double f10 = __ldg(p + ld), f11 = __ldg(p + ld + 1);
        const double lo = fma(wt, f01 - f00, f00);
        const double hi = fma(wt, f11 - f10, f10);
        v[k] = fma(wr, hi - lo, lo);
    }
}

// The same bilinear interpolant from per-cell coefficients: component k's
// cell (i, j) holds (a, b, c, d) = (f00, f10 - f00, f01 - f00,
// f11 - f10 - f01 + f00) at 4 (i ld + j) (r index first; built by k_field_coef
// before each push), so that f = a + b w_r + w_th (c + d w_r) is 3 FMA.  All in FP64,
// 26 operations a gather: the FP64 pipe has room beside the right-hand side's
// integer work.  With the weights and differences in paired FP32 (10 FP64
// operations, 230 issue slots more) a cell whose values differ as much as
// themselves was gathered to 4e-14 of them (now 8e-16), and a push was slower:
// 2^20 particles on 512^2 1006 -> 988 us, the batch of 12 runs 853 -> 782 us.
struct FieldsC {
    const double* c[6];
};

// Field tile staged in shared memory for a block of cell-sorted particles:
// STAGE_TI coefficient rows (r cells) x STAGE_TJ coefficient cells (th) of
// each of the six components, starting at coefficient cell (i0, j0).  A
// gather whose cell lies in the tile reads shared memory, any other the
// global coefficients (so staging never changes a result).
constexpr int STAGE_TI = 5, STAGE_TJ = 16;
struct StageTile {
    const double* s;    // shared: [6][STAGE_TI][4 * STAGE_TJ]; nullptr = nothing staged
    int i0, j0;
};

__device__ __forceinline__ double cell_value(double2 ab, double2 cd, double wr, double wt)
{
    return fma(wt, fma(cd.y, wr, cd.x), fma(ab.y, wr, ab.x));
}

// gather_c where an estimated cell is not the right one.
static __device__ __noinline__ void gather_far(const GridDev& G, const FieldsC& F, double r, double th, double v[6])
{
    const float lr = __logf(f32_cut(r));
    int at[4], mh;
    double w[4], tnv, thv;
    theta_views(G, th, tnv, thv, mh);
    locate(G.rn, G.irn, G.Nr + 1, r, (lr - G.lr0) * G.ilr, at[0], w[0]);
    locate(G.rh, G.irh, G.Nr, r, (lr - G.lrh0) * G.ilr, at[1], w[1]);
    locate(G.tn, G.itn, G.Nth + 1, tnv, (f32_cut(tnv) - G.t0) * G.it, at[2], w[2]);
    locate(G.th, G.ith, mh, thv, (f32_cut(thv) - G.th0) * G.it, at[3], w[3]);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const bool ro = (k == 0 || k == 4 || k == 5);
        const bool to = (k == 1 || k == 3 || k == 5);
        const double2* q = reinterpret_cast<const double2*>(F.c[k] + 4 * ((size_t)at[ro] * G.ld + at[2 + to]));
        v[k] = cell_value(__ldg(q), __ldg(q + 1), w[ro], w[2 + to]);
    }
}

template <bool STAGED = false>
__device__ __forceinline__ void gather_c(const GridDev& G, const FieldsC& F, double r, double th, double D[3], double B[3],
                                         const StageTile* T = nullptr)
{
    const float lr = __logf(f32_cut(r));
    double tnv, thv;
    int mh;
    theta_views(G, th, tnv, thv, mh);
    const float tfn = f32_cut(tnv), tfh = G.full ? f32_cut(thv) : tfn;
    int i0, i1, j0, j1;
    double wr0, wr1, wt0, wt1;
    locate_est(G.rn, G.irn, G.Nr + 1, r, (lr - G.lr0) * G.ilr, i0, wr0);
    locate_est(G.rh, G.irh, G.Nr, r, (lr - G.lrh0) * G.ilr, i1, wr1);
    locate_est(G.tn, G.itn, G.Nth + 1, tnv, (tfn - G.t0) * G.it, j0, wt0);
    locate_est(G.th, G.ith, mh, thv, (tfh - G.th0) * G.it, j1, wt1);
    const int ld = G.ld;
    double v[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const bool ro = (k == 0 || k == 4 || k == 5);
        const bool to = (k == 1 || k == 3 || k == 5);
        const int i = ro ? i1 : i0, j = to ? j1 : j0;
        const double wr = ro ? wr1 : wr0, wt = to ? wt1 : wt0;
        double2 ab, cd;
        const unsigned ti = STAGED ? (unsigned)(i - T->i0) : 0u, tj = STAGED ? (unsigned)(j - T->j0) : 0u;
        if (STAGED && T->s && ti < (unsigned)STAGE_TI && tj < (unsigned)STAGE_TJ) {
            const double2* q = reinterpret_cast<const double2*>(T->s + ((k * STAGE_TI + ti) * STAGE_TJ + tj) * 4);
            ab = q[0];
            cd = q[1];
        } else {
            const double2* q = reinterpret_cast<const double2*>(F.c[k] + 4 * ((size_t)i * ld + j));
            ab = __ldg(q);
            cd = __ldg(q + 1);
        }
        v[k] = cell_value(ab, cd, wr, wt);
    }
    // D^ph takes the weights of the nodes, B^ph those of the half nodes
    if (is_nan(v[2]) || is_nan(v[5])) {
        double u[6];
        gather_far(G, F, r, th, u);
#pragma unroll
        for (int k = 0; k < 6; ++k) v[k] = u[k];
    }
    D[0] = v[0]; D[1] = v[1]; D[2] = v[2];
    B[0] = v[3]; B[1] = v[4]; B[2] = v[5];
}

// What the Newton form of the implicit-midpoint solve needs from one
// right-hand side: u^i = g^ij u_j, 1 / Gamma, alpha / Gamma, g^ij, the
// magnetic-force factor qm alpha sqrt(gamma) / Gamma (0 without a field),
// B^i and u x B.
struct RhsJ {
    double U[3], iG, aiG;
    double gurr, gurp, gutt, gupp;
    double ks;
    double B[3], cx[3];
};

// Equations of motion at y (Eqs. p1, p2, O1, O2) and, as a by-product, the
// Hamiltonian H(y) = alpha Gamma - beta u_r - (q/m) A_0 (Eq. Ham with the
// Wald A_0 when B0pot != 0).  D, B: FIDO fields at y (ignored if !em).
// JAC: also fill *J (RhsJ) for the Newton iteration.
template <bool JAC>
__device__ __forceinline__ void eval_rhs_sc_t(const BH& bh, const double y[6], double s, double c, double qm,
                                              bool em, const double D[3], const double B[3], double B0pot,
                                              double f[6], double& H, RhsJ* J)
{
    const double r = y[0], ur = y[3], ut = y[4], up = y[5];
    // metric (App. A): e = xi - 1 = 2 M r / rho^2, beta^r = e / xi, g^rph = a / rho^2,
    // g^thth = 1 / rho^2, t = g^phph = 1 / (rho^2 sin^2 th)
    const double s2 = s * s, rho2 = fma(bh.a2, c * c, r * r);
    const double t = rcp_nr(rho2 * s2), irho2 = t * s2;
    const double mi = bh.twoM * irho2, e = mi * r, xi = fma(mi, r, 1.0);
    const double alpha = rsqrt_nr(xi), ixi = alpha * alpha, beta = e * ixi;
    const double gurp = bh.a * irho2, as2 = bh.a * s2;
    // u^i = g^ij u_j: u^r = u_r / xi + g^rph (a s^2 u_r + u_ph)
    const double g1 = fma(as2, ur, up), iu = ixi * ur, tu = t * up;
    const double Ur = fma(gurp, g1, iu), Ut = irho2 * ut, Up = fma(gurp, ur, tu);
    // W = a^2 s^2 u_r^2 + 2 a u_r u_ph + u_th^2, Q = W / rho^2 + u_ph^2 t, so that
    // Gamma^2 = 1 + u_r^2 / xi + Q
    const double W = fma(bh.a * ur, g1 + up, ut * ut);
    const double Q = fma(W, irho2, tu * up);
    const double G2 = fma(iu, ur, 1.0 + Q);
    const double iG = rsqrt_nr(G2);
    const double aiG = alpha * iG;
    f[0] = fma(aiG, Ur, -beta);
    f[1] = aiG * Ut;
    f[2] = aiG * Up;
    // du_i/dt = -Gamma d_i alpha + u_r d_i beta^r - (alpha / 2 Gamma) u_j u_k d_i g^jk
    // (Eq. p2).  With d alpha = -(alpha^3 / 2) d xi, d beta^r = d xi / xi^2,
    // d g^rr = a^2 s^2 d g^tt - d xi / xi^2 (+ q / rho^2 in th), d g^rp = a d g^tt
    // and q = 2 a^2 sin cos = -d_th rho^2:
    //   u_j u_k d_i g^jk = W d_i g^tt + u_ph^2 d_i g^pp - u_r^2 d_i xi / xi^2 (+ u_r^2 q / rho^2),
    // so the d_i xi factor is kap = (1/xi) ((u_r / xi)(1 + (alpha / Gamma) u_r / 2) +
    // alpha Gamma / 2), alpha Gamma = (alpha / Gamma) Gamma^2; k2 = 2 kap.
    //   r: d_r xi = (2 M / rho^2)(1 - 2 r^2 / rho^2), W d_r g^tt + u_ph^2 d_r g^pp
    //   = -2 (r / rho^2) Q;
    //   th: d_th g^tt = q / rho^4, d_th xi = e q / rho^2, d_th g^pp = -2 s c t^2 (rho^2 - a^2
    //   s^2), q / rho^2 = 2 a g^rph s c, so with P = W / rho^2 + u_r^2
    //   du_th/dt = a g^rph s c (2 e kap - (alpha / Gamma) P)
    //              + (alpha / Gamma) s c (t u_ph)^2 (rho^2 - a^2 s^2).
    const double GA = aiG * G2;                       // alpha Gamma
    const double k2 = ixi * fma(iu, fma(aiG, ur, 2.0), GA);
    const double rr = r * irho2;
    const double xk = mi * fma(-rr, r, 0.5);          // d_r xi / 2
    const double P = fma(W, irho2, ur * ur);
    const double br = fma(-aiG, P, e * k2), X2 = fma(-bh.a, as2, rho2);
    f[3] = aiG * rr;                                  // completed below
    f[4] = (s * c) * fma(aiG, (tu * tu) * X2, (bh.a * gurp) * br);
    f[5] = 0.0;
    double fr = 0.0;                                  // electromagnetic force in r
    if (JAC) {
        J->U[0] = Ur; J->U[1] = Ut; J->U[2] = Up;
        J->iG = iG; J->aiG = aiG;
        J->gurr = fma(bh.a * as2, irho2, ixi); J->gurp = gurp; J->gutt = irho2; J->gupp = t;
        // no field: the force terms of the Newton matrix vanish (set, not left undefined)
        J->ks = 0.0;
        J->B[0] = J->B[1] = J->B[2] = 0.0;
        J->cx[0] = J->cx[1] = J->cx[2] = 0.0;
    }
    if (em) {
        // (q/m) alpha gamma_ij D^j with gamma_rr = xi, gamma_rph = -a xi s^2,
        // gamma_thth = rho^2, gamma_phph = s^2 (rho^2 + a^2 xi s^2):
        //   r:  k xi X,  X = D^r - a s^2 D^ph
        //   ph: k s^2 (rho^2 D^ph - a xi X)
        const double k = qm * alpha;
        const double kr = k * rho2;
        const double ks = (qm * rho2) * (s * iG);    // k sqrt(gamma) / Gamma, alpha^2 xi = 1
        const double cr = fma(Ut, B[2], -Up * B[1]);
        const double ct = fma(Up, B[0], -Ur * B[2]);
        const double cp = fma(Ur, B[1], -Ut * B[0]);
        const double kx = (k * xi) * fma(-as2, D[2], D[0]);
        fr = fma(ks, cr, kx);
        f[4] = fma(kr, D[1], fma(ks, ct, f[4]));
        f[5] = fma(s2, fma(kr, D[2], -bh.a * kx), ks * cp);
        if (JAC) {
            J->ks = ks;
            J->B[0] = B[0]; J->B[1] = B[1]; J->B[2] = B[2];
            J->cx[0] = cr; J->cx[1] = ct; J->cx[2] = cp;
        }
    }
    f[3] = fma(f[3], Q, fma(xk, k2, fr));
    H = fma(-beta, ur, GA);                           // alpha Gamma - beta^r u_r
    if (not_zero(B0pot) && not_zero(qm)) {
        // A_0 = B0 a r (1 + cos^2 th) / rho^2   (Sec. 3.1.3)
        H = fma(-qm * B0pot * bh.a * r, fma(c, c, 1.0) * irho2, H);
    }
}

// eval_rhs_sc_t out of line, for the arguments rhs_x does not take.
template <bool JAC>
static __device__ __noinline__ void eval_rhs_call(const BH& bh, const double* y, double s, double c, double qm, bool em,
                                                  const double* D, const double* B, double B0pot, double* f, double& H,
                                                  RhsJ* J)
{
    eval_rhs_sc_t<JAC>(bh, y, s, c, qm, em, D, B, B0pot, f, H, J);
}

// The same right-hand side and H on integer mantissas of 60 bits (xf.cuh):
// results rounded once.  False, with nothing set, for what those do not
// carry: r not positive normal, s not normal (of either sign: half of the
// full-theta domain has sin th < 0), an infinity or a NaN among the arguments, a
// Gamma^2 that is not positive.
template <bool JAC = false>
FPIC_HD bool rhs_x(double bh_a, double bh_a2, double bh_twoM, const double y[6], double s, double c, double qm, bool em,
                   const double D[3], const double B[3], double B0pot, double f[6], double& H, bool want_F = true, bool want_H = true, RhsJ* J = nullptr)
{
    // exponent fields: r and s in 1 .. 2046, r positive, the others below 2047
    unsigned big = 0;
    {
        const double z[9] = {c, y[3], y[4], y[5], bh_a, bh_a2, bh_twoM, qm, B0pot};
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const unsigned h = (unsigned)(x_bits(z[i]) >> 32) & 0x7fffffffu;
            big = big > h ? big : h;
        }
        if (em) {
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                const unsigned h = (unsigned)(x_bits(i < 3 ? D[i] : B[i - 3]) >> 32) & 0x7fffffffu;
                big = big > h ? big : h;
            }
        }
        const unsigned hr = (unsigned)(x_bits(y[0]) >> 32), hs = (unsigned)(x_bits(s) >> 32) & 0x7fffffffu;
        if (big >= 0x7ff00000u || hr - 0x00100000u >= 0x7fe00000u || hs - 0x00100000u >= 0x7fe00000u) return false;
    }
    const xf r = x_from_pos(y[0]), sx = x_from(s), cx = x_from(c), ur = x_from(y[3]), ut = x_from(y[4]),
             up = x_from(y[5]);
    const xf a = x_from(bh_a), a2 = x_from(bh_a2), one = x_pow2(0);
    const xf s2 = x_sqr(sx), rho2 = x_norm(x_add(x_sqr(r), x_mul(a2, x_sqr(cx))));
    const xf t = x_rcp(x_mul(rho2, s2)), irho2 = x_norm(x_mul(t, s2));
    const xf mi = x_mul(x_from(bh_twoM), irho2), e = x_mul(mi, r), xi = x_norm(x_add(one, e));
    const xf alpha = x_rsqrt(xi), ixi = x_sqr(alpha), beta = x_mul(e, ixi);
    const xf gurp = x_mul(a, irho2), as2 = x_mul(a, s2);
    const xf g1 = x_norm(x_add(x_mul(as2, ur), up)), iu = x_mul(ixi, ur), tu = x_norm(x_mul(t, up));
    const xf Ur = x_add(x_mul(gurp, g1), iu), Ut = x_mul(irho2, ut), Up = x_add(x_mul(gurp, ur), tu);
    const xf W = x_norm(x_add(x_mul(x_mul(a, ur), x_add(g1, up)), x_sqr(ut))), Wi = x_mul(W, irho2);
    const xf Q = x_add(Wi, x_mul(tu, up)), G2 = x_norm(x_add(x_mul(iu, ur), x_add(one, Q)));
    if (G2.m <= 0) return false;
    const xf iG = x_rsqrt(G2), aiG = x_norm(x_mul(alpha, iG));
    if (JAC) {
        J->U[0] = x_to(Ur); J->U[1] = x_to(Ut); J->U[2] = x_to(Up);
        J->iG = x_to(iG); J->aiG = x_to(aiG);
        J->gurr = x_to(x_add(x_mul(x_mul(a, as2), irho2), ixi)); J->gurp = x_to(gurp);
        J->gutt = x_to(irho2); J->gupp = x_to(t);
        // no field: the force terms of the Newton matrix vanish (set, not left undefined)
        J->ks = 0.0;
        J->B[0] = J->B[1] = J->B[2] = 0.0;
        J->cx[0] = J->cx[1] = J->cx[2] = 0.0;
    }
    const xf GA = x_mul(aiG, G2);
    if (want_F) {
        f[0] = x_to(x_add(x_mul(aiG, Ur), x_neg(beta)));
        f[1] = x_to(x_mul(aiG, Ut));
        f[2] = x_to(x_mul(aiG, Up));
        const xf k2 = x_norm(x_mul(ixi, x_add(x_mul(iu, x_add(x_mul(aiG, ur), x_pow2(1))), GA)));
        const xf rr = x_mul(r, irho2), xk = x_mul(mi, x_add(x_pow2(-1), x_neg(x_mul(rr, r))));
        const xf P = x_add(Wi, x_sqr(ur)), br = x_add(x_mul(e, k2), x_neg(x_mul(aiG, P)));
        const xf X2 = x_add(rho2, x_neg(x_mul(a, as2)));
        xf f4 = x_mul(x_mul(sx, cx), x_add(x_mul(aiG, x_norm(x_mul(x_sqr(tu), X2))), x_mul(x_mul(a, gurp), br)));
        xf f3 = x_add(x_mul(x_mul(aiG, rr), Q), x_mul(xk, k2));
        f[5] = 0.0;
        if (em) {
            const xf q = x_from(qm), B0 = x_from(B[0]), B1 = x_from(B[1]), B2 = x_from(B[2]), D2 = x_from(D[2]);
            const xf k = x_mul(q, alpha), kr = x_mul(k, rho2), ks = x_norm(x_mul(x_mul(q, rho2), x_mul(sx, iG)));
            const xf cr = x_add(x_mul(Ut, B2), x_neg(x_mul(Up, B1))), ct = x_add(x_mul(Up, B0), x_neg(x_mul(Ur, B2))),
                     cp = x_add(x_mul(Ur, B1), x_neg(x_mul(Ut, B0)));
            if (JAC) {
                J->ks = x_to(ks);
                J->B[0] = B[0]; J->B[1] = B[1]; J->B[2] = B[2];
                J->cx[0] = x_to(cr); J->cx[1] = x_to(ct); J->cx[2] = x_to(cp);
            }
            const xf kx = x_mul(x_mul(k, xi), x_add(x_from(D[0]), x_neg(x_mul(as2, D2))));
            f3 = x_add3(f3, x_mul(ks, cr), kx);
            f4 = x_add3(f4, x_mul(kr, x_from(D[1])), x_mul(ks, ct));
            f[5] = x_to(x_add(x_mul(s2, x_add(x_mul(kr, D2), x_neg(x_mul(a, kx)))), x_mul(ks, cp)));
        }
        f[3] = x_to(f3);
        f[4] = x_to(f4);
    }
    if (want_H) {
        xf h = x_add(GA, x_neg(x_mul(beta, ur)));             // alpha Gamma - beta^r u_r
        if (x_bits(B0pot) << 1 && x_bits(qm) << 1)
            // A_0 = B0 a r (1 + cos^2 th) / rho^2   (Sec. 3.1.3)
            h = x_add(h, x_neg(x_mul(x_mul(x_mul(x_from(qm), x_from(B0pot)), x_mul(a, r)),
                                     x_mul(x_add(one, x_sqr(cx)), irho2))));
        H = x_to(h);
    }
    return true;
}

// Hamiltonian only (no derivatives, no force), given sin/cos of y[1].
__device__ __forceinline__ double eval_H_sc(const BH& bh, const double y[6], double s, double c, double qm,
                                            double B0pot)
{
    Geo g;
    geo_eval(bh, y[0], s, c, g);
    const double ur = y[3], ut = y[4], up = y[5];
    const double Ur = fma(g.gurr, ur, g.gurp * up);
    const double Ut = g.gutt * ut;
    const double Up = fma(g.gurp, ur, g.gupp * up);
    const double G = sqrt(fma(ur, Ur, fma(ut, Ut, fma(up, Up, 1.0))));
    double H = fma(g.alpha, G, -g.beta * ur);
    if (not_zero(B0pot) && not_zero(qm)) H = fma(-qm * B0pot * bh.a * y[0], fma(c, c, 1.0) * g.irho2, H);
    return H;
}

// The two parts of H at z (Sec. 3.1.2): kin = alpha Gamma - beta^r u_r and
// pot = (q/m) A_0 of the Wald potential (B0pot = 0: none); H = kin - pot and
// the error normaliser D0 = |kin| + |pot|.
__device__ __forceinline__ void h_parts(const BH& bh, const double z[6], double qm, double B0pot, double& kin,
                                        double& pot)
{
    double s, c;
    sincos(z[1], &s, &c);
    Geo g;
    geo_eval(bh, z[0], s, c, g);
    const double ur = z[3], ut = z[4], up = z[5];
    const double G2 = fma(ur, fma(g.gurr, ur, g.gurp * up),
                          fma(ut, g.gutt * ut, fma(up, fma(g.gurp, ur, g.gupp * up), 1.0)));
    kin = fma(g.alpha, sqrt(G2), -g.beta * ur);
    pot = 0.0;
    if (B0pot != 0.0 && qm != 0.0) pot = qm * B0pot * bh.a * z[0] * (1.0 + c * c) * g.irho2;
}

__device__ __forceinline__ double eval_H(const BH& bh, const double y[6], double qm, double B0pot)
{
    double s, c;
    sincos(y[1], &s, &c);
    return eval_H_sc(bh, y, s, c, qm, B0pot);
}

// The Wald field (App. B.1) at (r, th) with sin/cos of th given: B^i =
// eta^ijk d_j A_k / sqrt(gamma) from the potentials of Eq. (Amu), E_i =
// d_i A_0, D^i raised from Eq. (Ei) with beta = (beta^r, 0, 0).
__device__ __forceinline__ void wald_point_sc(const BH& bh, double B0, double r, double s, double c, double D[3],
                                              double B[3])
{
    Geo g;
    geo_eval(bh, r, s, c, g);
    const double M = bh.M, a = bh.a, a2 = bh.a2;
    const double P = g.rho2, iP = g.irho2, iP2 = iP * iP;
    const double sc = s * c, s2 = s * s, c2p1 = 1.0 + c * c;
    const double q = a2 * c2p1 - P;                 // enters d_th[(1+c^2)/rho^2]
    const double isg = 1.0 / g.sqrtg;
    const double dAph_t = B0 * sc * (r * r + a2 - 2.0 * M * a2 * r * c2p1 * iP - 2.0 * M * a2 * r * s2 * q * iP2);
    const double dAph_r = 0.5 * B0 * s2 * (2.0 * r - 2.0 * M * a2 * c2p1 * (P - 2.0 * r * r) * iP2);
    const double dAr_t = B0 * a * sc * (-1.0 + 2.0 * M * r * q * iP2);
    B[0] = dAph_t * isg;
    B[1] = -dAph_r * isg;
    B[2] = -dAr_t * isg;
    const double Er = B0 * a * M * c2p1 * (P - 2.0 * r * r) * iP2;
    const double Et = 2.0 * B0 * a * M * r * sc * q * iP2;
    // D_i from Eq. (Ei) with beta = (beta^r, 0, 0), then raised
    const double Dr_ = Er / g.alpha;
    const double Dt_ = (Et + g.sqrtg * g.beta * B[2]) / g.alpha;
    const double Dp_ = -g.sqrtg * g.beta * B[1] / g.alpha;
    D[0] = fma(g.gurr, Dr_, g.gurp * Dp_);
    D[1] = g.gutt * Dt_;
    D[2] = fma(g.gurp, Dr_, g.gupp * Dp_);
}

}  // namespace fpic
