"""The deposit on grids fine enough for the per-cell polynomials, against the
oracle's point-by-point quadrature."""
import numpy as np
import pytest

import oracle as O
from oracle import pic as P
from paper_2602_07452_gb300 import inputs as I
from helpers import cuda_or_skip, fpic, make_particles

pytestmark = pytest.mark.gpu


def _velocity(a, z):
    """Size of the FIDO velocity's terms: |v^i| with each of its terms taken
    absolutely (r and ph have two, which may cancel)."""
    r, th, u = z[:, 0], z[:, 1], z[:, 3:]
    s, c = np.sin(th), np.cos(th)
    P2 = r * r + a * a * c * c
    xi = 1.0 + 2.0 * r / P2
    t = [[(a * a * s * s / P2 + 1.0 / xi) * u[:, 0], a / P2 * u[:, 2]], [u[:, 1] / P2],
         [a / P2 * u[:, 0], u[:, 2] / (P2 * s * s)]]
    G = np.sqrt(1.0 + sum(sum(x) * u[:, i] for i, x in enumerate(t)))
    return [sum(np.abs(y) for y in x) / G for x in t]


@pytest.mark.parametrize("a,nr,nth,r_hi", [(0.0, 220, 230, 25.0), (0.9, 257, 301, 50.0), (0.99, 512, 222, 50.0),
                                           (0.99, 1024, 640, 50.0)])
def test_polynomial_deposit(a, nr, nth, r_hi):
    """30000 particles over the whole grid, a fifth of them in the cells at the
    poles and the horizon, some on nodes, half nodes and past the ends (held
    there).  A share is off by at most POLY_TOL = 2e-14 of the particle's
    charge and eight roundings of the paired arithmetic (2^-46): a node by
    1.4e-13 of the charge (or the current Q v) in the cells that touch it."""
    cuda_or_skip()
    F = fpic()
    g = I.log_grid(nr, nth, 0.9 * I.horizon(1.0, a), r_hi)
    ctx = F.fpic_init_metric(1.0, a)
    F.fpic_set_grid(ctx, g)
    n = 30000
    rng = np.random.default_rng(nr)
    d, q, _ = I.thermal_draws(n, g, 1.01 * I.horizon(1.0, a), g.rn[-1], 0.5, seed=nth)
    d[:2000, 1] = rng.uniform(0.2 * g.tn[0], g.tn[1], 2000)
    d[2000:4000, 1] = np.pi - rng.uniform(0.2 * g.tn[0], g.tn[1], 2000)
    d[4000:6000, 0] = rng.uniform(1.0001, 1.02, 2000) * I.horizon(1.0, a)
    lo = np.searchsorted(g.rn, 1.02 * I.horizon(1.0, a))
    d[6000:6100, 0] = g.rn[rng.integers(lo, nr + 1, 100)]
    d[6100:6200, 0] = g.rh[rng.integers(lo, nr, 100)]
    d[6200:6300, 1] = g.tn[rng.integers(0, nth + 1, 100)]
    d[6300:6400, 1] = g.th[rng.integers(0, nth, 100)]
    d[6400:6410, 0] = g.rn[-1]
    z = O.seed_fido(1.0, a, d)
    w = rng.uniform(0.5, 2.0, n)
    alive = (rng.random(n) > 0.05).astype(np.uint8)
    ref = [x.reshape(g.Nr + 1, g.ld) for x in P.deposit(1.0, a, g, z, q, w, alive)]
    p = make_particles(z, q, w=w, alive=alive)
    out = [t.cpu().numpy().reshape(g.Nr + 1, g.ld) for t in F.fpic_deposit(ctx, p, g.size)]
    # what a node's sum is divided by, from the oracle itself: a unit charge's shares add up to one
    cell = lambda X, x: np.clip(np.searchsorted(X, x, side="right") - 1, 0, len(X) - 2)
    v = _velocity(a, z)
    for k, (X, Y, amp) in enumerate(((g.rn, g.tn, 1.0), (g.rh, g.tn, v[0]), (g.rn, g.th, v[1]), (g.rn, g.tn, v[2]))):
        i, j = cell(X, z[:, 0]), cell(Y, z[:, 1])
        near = np.zeros((g.Nr + 1, g.ld))
        for di in (0, 1):
            for dj in (0, 1):
                np.add.at(near, (i + di, j + dj), np.abs(w * q * amp) * alive)
        m = (slice(0, len(X)), slice(0, len(Y)))
        vol = _dual(a, g, k in (1,), k in (2,))
        err = np.abs(out[k] - ref[k])[m] * vol
        assert err[near[m] == 0].size == 0 or err[near[m] == 0].max() == 0.0
        worst = (err[near[m] > 0] / near[m][near[m] > 0]).max()
        print("component", k, "worst node %.2e" % worst)
        assert worst <= 1.4e-13, (k, worst)


def _dual(a, g, ro, to):
    """2 pi x the trapezoid dual volume of the sub-grid's nodes."""
    e = lambda n, h, half: (n[:-1], n[1:]) if half else (np.r_[n[:1], h], np.r_[h, n[-1:]])
    x0, x1 = (x[:, None] for x in e(g.rn, g.rh, ro))
    y0, y1 = (x[None] for x in e(g.tn, g.th, to))
    acc, wt = 0.0, (0.5, 1.0, 1.0, 0.5)
    for ll in range(4):
        th = y0 + ll * (y1 - y0) / 3.0
        for kk in range(4):
            r = x0 + kk * (x1 - x0) / 3.0
            P2 = r * r + (a * np.cos(th)) ** 2
            acc = acc + wt[ll] * wt[kk] * np.sin(th) * np.sqrt(P2 * (P2 + 2.0 * r))
    return 2.0 * np.pi * acc * (x1 - x0) * (y1 - y0) / 9.0
