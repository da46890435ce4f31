"""Single node shares of the deposit, relative to themselves, on grids about the
lines between the lattices and the per-cell polynomials of degree 6 and 5."""
import numpy as np
import pytest

from paper_2602_07452_gb300 import inputs as I
from helpers import cuda_or_skip, fpic, make_particles

pytestmark = pytest.mark.gpu
L = np.longdouble


def _volume(a, x0, x1, y0, y1):
    acc, wt = L(0), (L(0.5), L(1), L(1), L(0.5))
    for k in range(4):
        x = x0 + k * (x1 - x0) / 3
        for m in range(4):
            y = y0 + m * (y1 - y0) / 3
            P = x * x + (a * np.cos(y)) ** 2
            acc = acc + wt[k] * wt[m] * np.sin(y) * np.sqrt(P * (P + 2 * x))
    return acc * (x1 - x0) * (y1 - y0) / 9


@pytest.mark.parametrize("a,side", [(0.5, 90), (0.5, 100), (0.9, 140), (0.9, 170), (0.9, 182), (0.99, 170),
                                    (0.99, 200), (0.99, 230), (0.99, 512)])
def test_small_shares_keep_their_relative_accuracy(a, side):
    """One unit charge in every ninth cell, so that a node holds one share:
    rho times the dual volume is that share.  Relative error of the shares down
    to 1e-6, corners and edges of the cells included: the square root's 4e-14 (the
    polynomials' bound, 1.3e-13 at most, is of the cells within the horizon, a
    fifth of it where these charges are) and eight roundings of the paired
    arithmetic (2^-46): 1.6e-13."""
    cuda_or_skip()
    F = fpic()
    g = I.log_grid(side, side, 0.9 * I.horizon(1.0, a), 50.0)
    ctx = F.fpic_init_metric(1.0, a)
    F.fpic_set_grid(ctx, g)
    rng = np.random.default_rng(side)
    lo = int(np.searchsorted(g.rn, 1.02 * I.horizon(1.0, a))) + 1
    i, j = (x.ravel() for x in np.meshgrid(np.arange(lo, side - 1, 3), np.arange(1, side - 1, 3), indexing="ij"))
    pick = rng.permutation(i.size)[:4000]
    i, j = i[pick], j[pick]
    n = i.size
    near = 0.5 * 10.0 ** rng.uniform(-6, 0, (2, n))
    kind = rng.integers(0, 3, (2, n))
    fr = np.choose(kind, [rng.random((2, n)), near, 1.0 - near])
    z = np.zeros((n, 6))
    z[:, 0] = g.rn[i] + fr[0] * (g.rn[i + 1] - g.rn[i])
    z[:, 1] = g.tn[j] + fr[1] * (g.tn[j + 1] - g.tn[j])
    rho = F.fpic_deposit(ctx, make_particles(z, np.ones(n)), g.size)[0].cpu().numpy().reshape(g.Nr + 1, g.ld)
    X, Y, x, y = g.rn.astype(L), g.tn.astype(L), z[:, 0].astype(L), z[:, 1].astype(L)
    V = {(b, d): _volume(L(a), X[i] if b else x, x if b else X[i + 1], Y[j] if d else y, y if d else Y[j + 1])
         for b in (0, 1) for d in (0, 1)}
    total = sum(V.values())
    two_pi = 2 * (L(np.pi) + L(1.2246467991473532e-16))
    for b in (0, 1):
        for d in (0, 1):
            share = V[b, d] / total
            got = rho[i + b, j + d] * two_pi * _volume(L(a), g.rh.astype(L)[i + b - 1], g.rh.astype(L)[i + b],
                                                       g.th.astype(L)[j + d - 1], g.th.astype(L)[j + d])
            m = share > 1e-6
            err = np.abs(got / share - 1)[m].astype(float)
            assert err.max() <= 1.6e-13, (b, d, err.max())
