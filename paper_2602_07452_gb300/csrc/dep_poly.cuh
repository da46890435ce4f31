// The deposit's subvolumes on fine grids from a per-cell polynomial of
// sqrt(gamma), in place of evaluating the trapezoid lattice point by point.
//
// On a sub-grid cell of centre (xm, yc) and size (dx, dy), with xi, eta in
// [-1/2, 1/2] its local coordinates,
//   sqrt(gamma) = K (sin th / sin yc) (1 + sum_{1 <= m+n <= DEG} f_mn xi^m eta^n),
// sqrt(gamma) / sin th = sqrt((r^2 + A)(r^2 + 2 M r + A)), A = a^2 cos^2 th.
// The 4-point trapezoid rule over an interval of centre u and half-width w
// is the mean over u + w {-1, -1/3, 1/3, 1} with weights {1, 2, 2, 1} / 6: its
// moments of xi^m are polynomials M_m(u, w) (mu_2 = 11/27, mu_4 = 83/243,
// mu_6 = 731/2187), so a subvolume is its area times
//   sum_n R_n E_n,  R_n = sum_m f_mn M_m (r part),  E_n the moments of
//   (sin th / sin yc) eta^n (th part; sin th by its own series about yc, so
//   the cells at the poles are no worse than the others).
// The same rule's values as the lattices' to the truncation at degree DEG = 5 or,
// on coarser grids, 6 and rounding: the terms up to degree 2 and everything they
// multiply run in paired FP32, the others (below 2^-20 of the sum where the table
// is used) in FP32.
#pragma once
#include <math.h>

#include "ff.cuh"

namespace fpic {

// floats of a cell (DEG 5: 25 used; 6: 32): seven or eight 16-byte loads
__host__ __device__ constexpr int poly_stride(int DEG)
{
    return DEG == 5 ? 28 : 32;
}

// A polynomial is used where poly_bound, the largest relative error of a node
// share over every cell of the grid (those inside the horizon too), stays below
// poly_tol: degree 5 if it does, else degree 6 (seven terms a cell and a paired
// one of E_1 more: 3 % of a deposit of 64 particles a cell on 140^2; the lattices
// take 1.8 times as long), else the lattices.  Grids uniform in ln r and th from 0.9 r_+ to
// 50 M take degree 5 from 150 (a = 0.5), 220 (0.9) or 275 (0.99) cells a side,
// degree 6 from 95, 140 or 170.  There a share down to 1e-6 is off by 5e-15 to 9e-15
// of itself (rms over a million; at most 1.1e-13), from the lattices by 1.1e-14
// (1.0e-13).
__host__ __device__ constexpr double poly_tol(int DEG)
{
    return DEG == 5 ? 4e-14 : 2.7e-14;
}
constexpr double POLY_MAX_DTH = 0.03, POLY_MAX_TAU = 4.0;     // limits of the sin th series

// What a th cell of centre yc (sin, cos given) and size dy brings to its cells'
// series: P1 = r^2 + a^2 cos^2 th = r^2 + sum_n p[n] eta^n.
template <int DEG>
struct PolyTheta {
    double p[DEG + 2];
};

template <int DEG>
__host__ __device__ inline void poly_theta(double a, double s, double c, double dy, PolyTheta<DEG>& t)
{
    const double s2y = 2.0 * s * c, c2y = 2.0 * c * c - 1.0;
    double h = 0.5 * a * a;
#pragma unroll
    for (int n = 1; n <= DEG + 1; ++n) {
        h *= 2.0 * dy * (1.0 / n);
        const double v = (n & 1) ? s2y : c2y;
        t.p[n] = ((n & 3) == 1 || (n & 3) == 2) ? -h * v : h * v;
    }
    t.p[0] = a * a * c * c;
}

// Coefficient (m, n) of g = P1 (P1 + 2 M r), P1 = x^2 + sum p[n] eta^n + p1 xi + p2 xi^2.
template <typename R>
__host__ __device__ inline R poly_g(int m, int n, const R* p, R p1, R p2, R q0, R q1)
{
    R g = R(0);
    if (m == 0) {
        g = q0 * p[n];
#pragma unroll
        for (int j = 0; j <= n; ++j) g += p[j] * p[n - j];
    } else if (m == 1) {
        g = (R(2) * p1 + q1) * p[n] + (n == 0 ? q0 * p1 : R(0));
    } else if (m == 2) {
        g = R(2) * p2 * p[n] + (n == 0 ? p1 * p1 + q0 * p2 + q1 * p1 : R(0));
    } else if (n == 0 && m == 3) {
        g = R(2) * p1 * p2 + q1 * p2;
    } else if (n == 0 && m == 4) {
        g = p2 * p2;
    }
    return g;
}

// f_mn of a cell of centre r = x and size dx: f = sqrt(g / g_00), to degree 3 in
// FP64 (f[m][n]), to degree DEG + 1 in FP32 (q): those terms are used in FP32 and,
// at degree DEG + 1, only bound the error.
template <int DEG>
__host__ __device__ inline void poly_series(double M, double x, double dx, const PolyTheta<DEG>& th, double f[4][4],
                                            float q[DEG + 2][DEG + 2])
{
    double p[DEG + 2];
#pragma unroll
    for (int n = 0; n < DEG + 2; ++n) p[n] = th.p[n];
    p[0] += x * x;
    const double p1 = 2.0 * x * dx, p2 = dx * dx, q0 = 2.0 * M * x, q1 = 2.0 * M * dx;
    const double ig = 1.0 / (p[0] * (p[0] + q0));
#pragma unroll
    for (int d = 0; d <= 3; ++d)
#pragma unroll
        for (int m = 0; m <= d; ++m) {
            const int n = d - m;
            double t = poly_g<double>(m, n, p, p1, p2, q0, q1) * ig;
#pragma unroll
            for (int i = 0; i <= m; ++i)
#pragma unroll
                for (int j = 0; j <= n; ++j)
                    if (i + j > 0 && i + j < d) t -= f[i][j] * f[m - i][n - j];
            f[m][n] = d == 0 ? 1.0 : 0.5 * t;
            q[m][n] = (float)f[m][n];
        }
    // normalized by g_00 = (1 / ig): the float factors stay in range
    const double is = sqrt(ig);
    float pf[DEG + 2];
#pragma unroll
    for (int n = 0; n < DEG + 2; ++n) pf[n] = (float)(p[n] * is);
    const float p1f = (float)(p1 * is), p2f = (float)(p2 * is), q0f = (float)(q0 * is), q1f = (float)(q1 * is);
#pragma unroll
    for (int d = 4; d <= DEG + 1; ++d)
#pragma unroll
        for (int m = 0; m <= d; ++m) {
            const int n = d - m;
            float t = poly_g<float>(m, n, pf, p1f, p2f, q0f, q1f);
#pragma unroll
            for (int i = 0; i <= m; ++i)
#pragma unroll
                for (int j = 0; j <= n; ++j)
                    if (i + j > 0 && i + j < d) t -= q[i][j] * q[m - i][n - j];
            q[m][n] = 0.5f * t;
        }
}

// Bound on the relative error of a node share: the terms of degree DEG + 1 that
// are left out and the FP32 rounding of those of degree 3 to DEG, at the cell's
// corners (where the interval of a small share lies).
template <int DEG>
__host__ __device__ inline float poly_bound(const float f[DEG + 2][DEG + 2])
{
    float e = 0.f;
#pragma unroll
    for (int d = 3; d <= DEG + 1; ++d)
#pragma unroll
        for (int m = 0; m <= d; ++m)
            e += fabsf(f[m][d - m]) * (d == DEG + 1 ? 1.f : 5.9604644775390625e-8f) / (float)(1 << d);
    return e;
}

// The larger of two bounds, b possibly a NaN (a series past the range of its
// numbers): infinite then, above every tolerance.
__host__ __device__ inline float poly_worst(float e, float b)
{
    if (!(b <= 3.402823466e38f)) return HUGE_VALF;
    return b > e ? b : e;
}

struct PolyTab {
    double lo[4], hi[4];    // first and last rn, rh, tn, th
    const float4* c[3];     // cells of the (i, j), (i+1/2, j), (i, j+1/2) sub-grids, row stride Nth
    const float2* ir[2];    // 1 / dr of the integer and half r cells
    const float4* t[2];     // two per integer and half th cell: 1 / dth and tau = dth cot yc (pairs);
                            // dth^2 / 2 and dth^2 / 6 (pairs)
};

#ifdef __CUDACC__
// One interval's moments: [0] below the particle, [1] above it.
struct Mom {
    ff len, m1, m2, m3;
    float m4, m5, m6, m7;
};

// Both intervals of a cell split at the fraction al (ab = 1 - al): lower
// u = -ab/2, w = al/2; upper u = al/2, w = ab/2.
__device__ __forceinline__ void moments(ff al, ff ab, Mom M[2])
{
    const ff mu2 = {__uint_as_float(0x3ed097b4u), __uint_as_float(0x3197b426u)};     // 11/27
    const ff a2 = ff_sqr(al), b2 = ff_sqr(ab);
    const ff ma = ff_mul(mu2, a2), mb = ff_mul(mu2, b2);
    constexpr float k6 = 22.f / 9.f, k10 = 110.f / 27.f, m4 = 83.f / 243.f, k5 = 415.f / 243.f, k15 = 165.f / 27.f,
                    k15b = 1245.f / 243.f, m6 = 731.f / 2187.f, k21 = 231.f / 27.f, k35 = 2905.f / 243.f,
                    k7 = 5117.f / 2187.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const ff U2 = h ? a2 : b2, W = h ? mb : ma;
        M[h].len = h ? ab : al;
        M[h].m1 = h ? ff_scale(al, 0.5f) : ff_scale(ab, -0.5f);
        M[h].m2 = ff_scale(ff_add(U2, W), 0.25f);
        M[h].m3 = ff_mul(M[h].m1, ff_scale(ff_add(U2, ff_mulf(W, 3.f)), 0.25f));
        const float u = M[h].m1.hi, u2 = 0.25f * U2.hi, w2 = 0.25f * (h ? b2 : a2).hi;
        const float uu = u2 * u2, uw = u2 * w2, ww = w2 * w2;
        M[h].m4 = fmaf(m4, ww, fmaf(k6, uw, uu));
        M[h].m5 = u * fmaf(k5, ww, fmaf(k10, uw, uu));
        M[h].m6 = fmaf(u2, fmaf(k15b, ww, fmaf(k15, uw, uu)), m6 * ww * w2);
        M[h].m7 = u * fmaf(u2, fmaf(k35, ww, fmaf(k21, uw, uu)), k7 * ww * w2);
    }
}

// th moments of (sin th / sin yc) eta^n: E_0 = 1 + e0.
struct MomT {
    ff len, e0, e1, e2;
    float e3, e4, e5, e6;
};

__device__ __forceinline__ ff ff_addf(ff a, float b)      // a + b, |b| far below |a| or folded into lo
{
    return {a.hi, __fadd_rn(a.lo, b)};
}

// d2_2, d2_6: dth^2 / 2 and dth^2 / 6.  The cubic term of sin th, up to 10^-6
// of the sum in the cells at the poles, is paired too; on coarser grids (DEG 6) so
// is E_1's term of dth^2.
template <int DEG>
__device__ __forceinline__ void moments_th(const Mom M[2], ff tau, ff d2_2, ff d2_6, MomT E[2])
{
    const float t = tau.hi, d = 2.f * d2_2.hi;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const Mom& m = M[h];
        E[h].len = m.len;
        // 1 - d^2/2 + d^4/24 and tau (1 - d^2/6 + d^4/120) in powers of eta
        const float c0 = d * d * fmaf(t * (1.f / 120.f), m.m5, (1.f / 24.f) * m.m4);
        const ff s1 = ff_mul(tau, ff_add(m.m1, ff_neg(ff_mul(d2_6, m.m3))));
        E[h].e0 = ff_addf(ff_add(s1, ff_neg(ff_mul(d2_2, m.m2))), c0);
        const float c1 = -d * fmaf(-d, fmaf((1.f / 120.f) * t, m.m6, (1.f / 24.f) * m.m5),
                                   DEG > 5 ? (1.f / 6.f) * t * m.m4 : fmaf((1.f / 6.f) * t, m.m4, 0.5f * m.m3.hi));
        ff e1 = ff_add(m.m1, ff_mul(tau, m.m2));
        if (DEG > 5) e1 = ff_add(e1, ff_neg(ff_mul(d2_2, m.m3)));
        E[h].e1 = ff_addf(e1, c1);
        const float c2 = -d * fmaf((1.f / 6.f) * t, m.m5, 0.5f * m.m4);
        E[h].e2 = ff_addf(ff_add(m.m2, ff_mul(tau, m.m3)), c2);
        E[h].e3 = fmaf(-d, fmaf((1.f / 6.f) * t, m.m6, 0.5f * m.m5), fmaf(t, m.m4, m.m3.hi));
        E[h].e4 = fmaf(-0.5f * d, m.m6, fmaf(t, m.m5, m.m4));
        E[h].e5 = fmaf(t, m.m6, m.m5);
        E[h].e6 = fmaf(t, m.m7, m.m6);
    }
}

// The four node shares (w00, w10, w01, w11: V of the opposite corner / V) of
// a sub-grid cell from its r and th moments.
template <int DEG>
__device__ __forceinline__ void poly_shares(const float4* __restrict__ c, const Mom X[2], const MomT Y[2], ff w[4])
{
    const float4 q0 = __ldg(c), q1 = __ldg(c + 1), q2 = __ldg(c + 2), q3 = __ldg(c + 3), q4 = __ldg(c + 4),
                 q5 = __ldg(c + 5);
    const float4 q6 = DEG > 5 ? __ldg(c + 6) : make_float4(__ldg((const float*)(c + 6)), 0.f, 0.f, 0.f);
    const float4 q7 = DEG > 5 ? __ldg(c + 7) : make_float4(0.f, 0.f, 0.f, 0.f);
    const ff f10 = {q0.x, q0.y}, f01 = {q0.z, q0.w}, f20 = {q1.x, q1.y}, f11 = {q1.z, q1.w}, f02 = {q2.x, q2.y};
    const float f30 = q2.z, f21 = q2.w, f12 = q3.x, f03 = q3.y, f40 = q3.z, f31 = q3.w, f22 = q4.x, f13 = q4.y,
                f04 = q4.z, f50 = q4.w, f41 = q5.x, f32 = q5.y, f23 = q5.z, f14 = q5.w, f05 = q6.x, f60 = q6.y,
                f51 = q6.z, f42 = q6.w, f33 = q7.x, f24 = q7.y, f15 = q7.z, f06 = q7.w;
    ff V[4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const Mom& m = X[h];
        constexpr bool six = DEG > 5;
        const float r0 = six ? fmaf(f60, m.m6, f50 * m.m5) : f50 * m.m5;
        const float r1 = six ? fmaf(f51, m.m5, f41 * m.m4) : f41 * m.m4;
        const float r2 = six ? fmaf(f42, m.m4, f32 * m.m3.hi) : f32 * m.m3.hi;
        const float r3 = six ? fmaf(f33, m.m3.hi, f03) : f03, r4 = six ? fmaf(f24, m.m2.hi, f04) : f04;
        const ff R0 = ff_addf(ff_add(ff_mul(f10, m.m1), ff_mul(f20, m.m2)), fmaf(f30, m.m3.hi, fmaf(f40, m.m4, r0)));
        const ff R1 = ff_addf(ff_add(f01, ff_mul(f11, m.m1)), fmaf(f21, m.m2.hi, fmaf(f31, m.m3.hi, r1)));
        const ff R2 = ff_addf(f02, fmaf(f12, m.m1.hi, fmaf(f22, m.m2.hi, r2)));
        const float R3 = fmaf(f13, m.m1.hi, fmaf(f23, m.m2.hi, r3)), R4 = fmaf(f14, m.m1.hi, r4),
                    R5 = six ? fmaf(f15, m.m1.hi, f05) : f05;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const MomT& e = Y[g];
            // sum - 1 = e0 + R0 + R0 e0 + R1 e1 + R2 e2 + ...
            ff S = ff_add(ff_add(e.e0, R0), ff_add(ff_mul(R0, e.e0), ff_mul(R1, e.e1)));
            // the low floats of R_1, E_1, R_2, E_2 carry FP32 terms of their own, far above
            // 2^-24 of the high ones: their products, which ff_mul leaves out, count
            // (up to 10^-12 of the sum on grids of 150 cells a side)
            const float h5 = six ? fmaf(R5, e.e5, f06 * e.e6) : R5 * e.e5;
            const float ll = fmaf(R1.lo, e.e1.lo, fmaf(R2.lo, e.e2.lo, h5));
            S = ff_add(S, ff_addf(ff_mul(R2, e.e2), fmaf(R3, e.e3, fmaf(R4, e.e4, ll))));
            const ff area = ff_mul(m.len, e.len);
            const ff v = ff_add(area, ff_mul(area, S));
            V[h + 2 * g] = ff_fast2(v.hi, v.lo);         // normalized: S carries FP32 terms in its lo
        }
    }
    const ff iV = ff_rcp(ff_add(ff_add(V[0], V[1]), ff_add(V[2], V[3])));
    w[0] = ff_mul(V[3], iV);
    w[1] = ff_mul(V[2], iV);
    w[2] = ff_mul(V[1], iV);
    w[3] = ff_mul(V[0], iV);
}
#endif

}  // namespace fpic
