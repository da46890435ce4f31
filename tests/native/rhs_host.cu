// rhs_x on the host against the same formulas in long double and in double:
// prints, per output, the L2 relative errors of both over random draws.
#include <cmath>
#include <cstdio>
#include <random>

#include "fpic_device.cuh"

using namespace fpic;

template <class T>
static void formulas(T a, const double* y, T s, T c, T qm, bool em, const double* D, const double* B, T B0, T f[7])
{
    const T r = y[0], ur = y[3], ut = y[4], up = y[5], s2 = s * s, rho2 = a * a * c * c + r * r, t = 1 / (rho2 * s2);
    const T ir = t * s2, mi = 2 * ir, e = mi * r, xi = 1 + e, al = 1 / std::sqrt(xi), ixi = al * al, beta = e * ixi;
    const T gurp = a * ir, as2 = a * s2, g1 = as2 * ur + up, iu = ixi * ur, tu = t * up;
    const T Ur = gurp * g1 + iu, Ut = ir * ut, Up = gurp * ur + tu, W = a * ur * (g1 + up) + ut * ut, Q = W * ir + tu * up;
    const T G2 = iu * ur + 1 + Q, iG = 1 / std::sqrt(G2), aiG = al * iG, GA = aiG * G2;
    const T k2 = ixi * (iu * (aiG * ur + 2) + GA), rr = r * ir, xk = mi * (T(0.5) - rr * r), P = W * ir + ur * ur;
    const T br = e * k2 - aiG * P, X2 = rho2 - a * as2;
    f[0] = aiG * Ur - beta;
    f[1] = aiG * Ut;
    f[2] = aiG * Up;
    f[3] = aiG * rr * Q + xk * k2;
    f[4] = s * c * (aiG * (tu * tu) * X2 + a * gurp * br);
    f[5] = 0;
    if (em) {
        const T k = qm * al, kr = k * rho2, ks = qm * rho2 * (s * iG), kx = k * xi * (D[0] - as2 * D[2]);
        f[3] += ks * (Ut * B[2] - Up * B[1]) + kx;
        f[4] += kr * D[1] + ks * (Up * B[0] - Ur * B[2]);
        f[5] = s2 * (kr * D[2] - a * kx) + ks * (Ur * B[1] - Ut * B[0]);
    }
    f[6] = GA - beta * ur - qm * B0 * a * r * (1 + c * c) * ir;
}

int main()
{
    std::mt19937_64 g(1);
    auto U = [&](double lo, double hi) { return lo + (hi - lo) * std::uniform_real_distribution<double>()(g); };
    for (int mode = 0; mode < 6; ++mode) {   // neutral; charged; a = 0, zeros; wide u; far and uneven fields; near the axis
        double ex[7] = {0}, ed[7] = {0}, n2[7] = {0};
        for (int it = 0; it < 40000; ++it) {
            const bool em = mode != 0;
            const double a = mode == 2 ? 0 : U(0, .999), qm = mode == 0 ? 0 : (mode == 3 ? U(-1e3, 1e3) : U(-10, 10));
            double y[6] = {mode == 4 ? std::exp(U(0, 9)) : U(1.1, 30), mode == 5 ? std::exp(U(-12, 0)) : U(.01, 3.13), 0};
            double D[3], B[3], f[6], H, fd[7];
            const double us = mode == 3 ? std::exp(U(-10, 10)) : 3, B0 = U(-1, 1);
            for (int i = 0; i < 3; ++i) {
                y[3 + i] = U(-us, us);
                D[i] = U(-1, 1) * (mode == 4 ? std::exp(U(-30, 5)) : 1);
                B[i] = U(-1, 1) * (mode == 4 ? std::exp(U(-30, 5)) : 1);
            }
            if (mode == 2 && it % 3 == 0) y[3 + it % 9 / 3] = B[it % 2] = 0;
            const double s = std::sin(y[1]), c = std::cos(y[1]);
            long double fl[7];
            formulas<long double>(a, y, s, c, qm, em, D, B, B0, fl);
            formulas<double>(a, y, s, c, qm, em, D, B, B0, fd);
            if (!rhs_x(a, a * a, 2.0, y, s, c, qm, em, D, B, B0, f, H)) return 1;
            for (int i = 0; i < 7; ++i) {
                const double x = (double)((i < 6 ? f[i] : H) - fl[i]), d = (double)(fd[i] - fl[i]), v = (double)fl[i];
                ex[i] += x * x;
                ed[i] += d * d;
                n2[i] += v * v;
            }
        }
        for (int i = 0; i < 7; ++i)
            std::printf("%d %d %.3e %.3e\n", mode, i, std::sqrt(ex[i] / (n2[i] + 1e-300)), std::sqrt(ed[i] / (n2[i] + 1e-300)));
    }
    // what it refuses: no mantissa in a factor, r or s not positive normal
    const double v[3] = {0.1, 0.2, 0.3}, bad[4] = {NAN, INFINITY, -INFINITY, 1e-310};
    double f[6], H;
    for (int k = 0; k < 4; ++k)
        for (int w = 0; w < 7; ++w) {
            double y[6] = {5, 1, 0, .1, .2, .3}, D[3] = {v[0], v[1], v[2]}, B[3] = {v[0], v[1], v[2]}, s = std::sin(1.0), q = 1;
            (w == 0 ? y[0] : w == 1 ? y[3] : w == 2 ? D[0] : w == 3 ? B[2] : w == 4 ? s : w == 5 ? q : y[5]) = bad[k];
            const bool want = k == 3 && w != 0 && w != 4;       // a subnormal counts as zero but in r and s
            if (rhs_x(.9, .81, 2.0, y, s, std::cos(1.0), q, true, D, B, 0.0, f, H) != want) return 2;
        }
    return 0;
}
