"""Rounding of the conserving deposit's cell sums."""
import numpy as np
import pytest

from paper_2602_07452_gb300 import inputs as I
from helpers import cuda_or_skip, fpic, make_particles

pytestmark = pytest.mark.gpu
L = np.longdouble


def test_sums_of_crowded_cells():
    """4096 resting charges of one sign in each of 144 cells apart: rho at their
    nodes against extended precision.  An addition is off by 0.29 x 1.5 x 2^-53 of
    its sum (uniform in half an ulp, the ulp's mean), a chain of m that grows
    evenly by 0.58 sqrt(m) times that: 128 groups one after the other and a group's
    five, twice (a row's two lanes, each half the sum): 2.3e-16 rms; four roundings
    of the normalisation 1e-16.  Held to twice that (a chain of 2048 has 9e-16)."""
    cuda_or_skip()
    F = fpic()
    a, per = 0.9, 4096
    g = I.log_grid(40, 40, 1.5, 20.0)
    ctx = F.fpic_init_metric(1.0, a)
    F.fpic_set_grid(ctx, g)
    i, j = (x.ravel() for x in np.meshgrid(np.arange(2, 38, 3), np.arange(2, 38, 3), indexing="ij"))
    rng = np.random.default_rng(4)
    ii, jj = np.repeat(i, per), np.repeat(j, per)
    n = ii.size
    z = np.zeros((n, 6))
    z[:, 0] = g.rn[ii] + rng.uniform(0.01, 0.99, n) * (g.rn[ii + 1] - g.rn[ii])
    z[:, 1] = g.tn[jj] + rng.uniform(0.01, 0.99, n) * (g.tn[jj + 1] - g.tn[jj])
    w = rng.uniform(0.5, 2.0, n)
    p = make_particles(z, np.ones(n), w=w)
    rho = F.fpic_deposit_conserving(ctx, p, p, 1e-3)[0].cpu().numpy().reshape(g.Nr + 1, g.ld)
    X, Y = g.rn.astype(L), g.tn.astype(L)
    x = (z[:, 0] - X[ii]) / (X[ii + 1] - X[ii])
    y = (z[:, 1] - Y[jj]) / (Y[jj + 1] - Y[jj])
    two_pi = 2 * (L(np.pi) + L(1.2246467991473532e-16))
    H, T = g.rh.astype(L), g.th.astype(L)
    err = []
    for b in (0, 1):
        for d in (0, 1):
            q = (w * (x if b else 1 - x) * (y if d else 1 - y)).reshape(-1, per).sum(1)
            s, c = np.sin(Y[j + d]), np.cos(Y[j + d])
            P = X[i + b] ** 2 + (L(a) * c) ** 2
            vol = two_pi * P * np.sqrt(1 + 2 * X[i + b] / P) * s * (H[i + b] - H[i + b - 1]) * (T[j + d] - T[j + d - 1])
            err.append((rho[i + b, j + d] * vol / q - 1).astype(float))
    rms = np.sqrt(np.mean(np.square(err)))
    print("rms %.2e" % rms)
    assert rms <= 5e-16, rms
