"""Rounding of the cell sums of the polynomial deposit."""
import numpy as np
import pytest

from paper_2602_07452_gb300 import inputs as I
from helpers import cuda_or_skip, fpic, make_particles

pytestmark = pytest.mark.gpu


def test_sums_of_equal_shares():
    """16384 equal charges at one place in each of 225 cells apart, against 16384
    times one such charge.  Additions of equal terms err to the same side while
    the sum stays in a binade: a chain of m by up to m/2 half ulps of a term.  The
    high floats' sums are chains of n / 8 in FP64, 2048 x 2^-54; the low ones' of 16
    in FP32, 2^-25 of the share: 16 x 2^-25 x 2^-25 at most: 1.3e-13."""
    cuda_or_skip()
    F = fpic()
    a, n, side = 0.9, 16384, 200
    g = I.log_grid(side, side, 0.9 * I.horizon(1.0, a), 50.0)
    ctx = F.fpic_init_metric(1.0, a)
    F.fpic_set_grid(ctx, g)
    rng = np.random.default_rng(8)
    i, j = (x.ravel() for x in np.meshgrid(np.arange(30, 180, 10), np.arange(20, 170, 10), indexing="ij"))
    z = np.zeros((i.size, 6))
    z[:, 0] = g.rn[i] + rng.uniform(0.05, 0.95, i.size) * (g.rn[i + 1] - g.rn[i])
    z[:, 1] = g.tn[j] + rng.uniform(0.05, 0.95, i.size) * (g.tn[j + 1] - g.tn[j])
    w = rng.uniform(0.5, 2.0, i.size)
    dep = lambda k: F.fpic_deposit(ctx, make_particles(np.repeat(z, k, 0), np.ones(i.size * k), w=np.repeat(w, k)),
                                   g.size)[0].cpu().numpy()
    one, many = dep(1), dep(n)
    at = one != 0
    assert at.sum() == 4 * i.size
    err = np.abs(many[at] / (n * one[at]) - 1.0)
    print("max %.2e" % err.max())
    assert err.max() <= 1.3e-13, err.max()
