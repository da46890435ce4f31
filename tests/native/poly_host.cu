// The per-cell polynomials' bound on the host: over rows of cells from a radius
// where the series is finite to one past its numbers' range, in either order.
#include <cstdio>

#include "dep_poly.cuh"

using namespace fpic;

static float row(double r)
{
    PolyTheta th;
    double f[4][4];
    float q[7][7];
    poly_theta(0.9, sin(1.0), cos(1.0), 0.01, th);
    poly_series(1.0, r, 0.01 * r, th, f, q);
    return poly_bound(q);
}

int main()
{
    const float near = row(2.0), far = row(1e85);
    std::printf("%d %d %d %d\n", near <= POLY_TOL, far != far, poly_worst(near, far) <= POLY_TOL,
                poly_worst(poly_worst(0.f, far), near) <= POLY_TOL);
    return 0;
}
