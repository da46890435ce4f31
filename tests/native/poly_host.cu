// The per-cell polynomials' bound on the host: over rows of cells from a radius
// where the series is finite to one past its numbers' range, in either order.
#include <cstdio>

#include "dep_poly.cuh"

using namespace fpic;

template <int DEG>
static float row(double r)
{
    PolyTheta<DEG> th;
    double f[4][4];
    float q[DEG + 2][DEG + 2];
    poly_theta<DEG>(0.9, sin(1.0), cos(1.0), 0.01, th);
    poly_series<DEG>(1.0, r, 0.01 * r, th, f, q);
    return poly_bound<DEG>(q);
}

template <int DEG>
static void check()
{
    const float near = row<DEG>(2.0), far = row<DEG>(1e85);
    std::printf("%d %d %d %d\n", near <= poly_tol(DEG), far != far, poly_worst(near, far) <= poly_tol(DEG),
                poly_worst(poly_worst(0.f, far), near) <= poly_tol(DEG));
}

int main()
{
    check<5>();
    check<6>();
    return 0;
}
