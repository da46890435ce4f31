// rhs_x on the host below the axis (th in (pi, 2 pi), sin th < 0): the mirror
// image of the state, with u_th, D^th, B^th of the other sign, has the same
// right-hand side but for that sign of its th components.
#include <cmath>
#include <cstdio>
#include <random>

#include "fpic_device.cuh"

using namespace fpic;

int main()
{
    std::mt19937_64 g(3);
    auto U = [&](double lo, double hi) { return lo + (hi - lo) * std::uniform_real_distribution<double>()(g); };
    double worst = 0;
    for (int it = 0; it < 100000; ++it) {
        const bool em = it & 1;
        const double a = U(0, .999), qm = U(-10, 10), th = it % 5 ? U(.01, 3.13) : std::exp(U(-12, 0)), B0 = U(-1, 1);
        double y[6] = {U(1.1, 30), th, 0, U(-3, 3), U(-3, 3), U(-3, 3)}, D[3], B[3], f[6], H, fm[6], Hm;
        for (int i = 0; i < 3; ++i) {
            D[i] = U(-1, 1);
            B[i] = U(-1, 1);
        }
        const double s = std::sin(th), c = std::cos(th);
        if (!rhs_x(a, a * a, 2.0, y, s, c, qm, em, D, B, B0, f, H)) return 1;
        y[4] = -y[4];
        D[1] = -D[1];
        B[1] = -B[1];
        if (!rhs_x(a, a * a, 2.0, y, -s, c, qm, em, D, B, B0, fm, Hm)) return 2;
        // each term within a unit or two of 2^-60 of its image, then one rounding;
        // the force's terms are of the size of q/m rho^2 and may cancel
        const double big = std::fabs(f[3]) + std::fabs(f[4]) + std::fabs(f[5]) + 1 +
                           (em ? 4 * std::fabs(qm) * (y[0] * y[0] + 1) : 0);
        for (int i = 0; i < 6; ++i)
            worst = std::fmax(worst, std::fabs(f[i] - (i == 1 || i == 4 ? -fm[i] : fm[i])) / (i < 3 ? 1 + std::fabs(f[i]) : big));
        worst = std::fmax(worst, std::fabs(H - Hm) / (1 + std::fabs(H)));
    }
    std::printf("%.3e\n", worst);
    return 0;
}
