"""The push's field gather against extended precision, on coarse and fine grids,
at field sizes far from one and on nodes its index estimate misses."""
import numpy as np
import pytest

from paper_2602_07452_gb300 import inputs as I
from helpers import cuda_or_skip, dev, fpic, make_particles

pytestmark = pytest.mark.gpu
L = np.longdouble


@pytest.mark.parametrize("side,scale,clustered", [(6, 1.0, False), (24, 1.0, False), (48, 1e-60, False),
                                                  (100, 1e40, False), (1000, 1.0, False), (60, 1.0, True)])
def test_gathered_force_of_a_rough_field(side, scale, clustered):
    """A random field (a cell's values differ as much as themselves), a = 0, a step
    of 2^-66 over which no state moves: u_ph / dt is q/m alpha (r sin th)^2 D^ph.
    Off by at most 2e-15 of the cell's largest value: three roundings of each
    weight and of its difference of up to twice that value, three of the
    interpolant's sums, five of the force's factors and sums (18 x 2^-53)."""
    cuda_or_skip()
    F = fpic()
    g = I.log_grid(side, side + 1, 1.9, 30.0)
    if clustered:
        t = np.linspace(0.0, 1.0, g.Nth + 1)
        g.tn = g.tn[0] + (g.tn[-1] - g.tn[0]) * (0.2 * t + 0.8 * t**3)
        g.th = 0.5 * (g.tn[:-1] + g.tn[1:])
        g.rn = 1.9 + 28.1 * np.linspace(0.0, 1.0, g.Nr + 1) ** 1.5
        g.rh = 0.5 * (g.rn[:-1] + g.rn[1:])
    ctx = F.fpic_init_metric(1.0, 0.0)
    F.fpic_set_grid(ctx, g)
    rng = np.random.default_rng(side)
    f = [np.zeros(g.size) for _ in range(6)]
    f[2] = rng.normal(size=g.size) * scale
    n, dt = 20000, 2.0**-66
    r = np.exp(rng.uniform(np.log(2.05), np.log(29.5), n))
    th = rng.uniform(1.01 * g.tn[0], 0.999 * g.tn[-1], n)
    z = np.zeros((n, 6))
    z[:, 0], z[:, 1] = r, th
    p = make_particles(z, np.full(n, 1.0 / scale), H0=np.ones(n), D0=np.ones(n), Hn=np.ones(n))
    F.fpic_push(ctx, p, [dev(x) for x in f], F.push_params(dt, scheme=F.FPIC_RK4))
    got = p.uph.cpu().numpy() / dt
    X, Y, q = g.rn.astype(L), g.tn.astype(L), f[2].reshape(g.Nr + 1, g.ld).astype(L)
    i = np.clip(np.searchsorted(g.rn, r, side="right") - 1, 0, g.Nr - 1)
    j = np.clip(np.searchsorted(g.tn, th, side="right") - 1, 0, g.Nth - 1)
    x, y = (r - X[i]) / (X[i + 1] - X[i]), (th - Y[j]) / (Y[j + 1] - Y[j])
    want = (1 - x) * ((1 - y) * q[i, j] + y * q[i, j + 1]) + x * ((1 - y) * q[i + 1, j] + y * q[i + 1, j + 1])
    size = L(1.0 / scale) / np.sqrt(1 + 2 / r.astype(L)) * (r * np.sin(th.astype(L))) ** 2
    big = np.abs(np.stack([q[i, j], q[i + 1, j], q[i, j + 1], q[i + 1, j + 1]])).max(0)
    err = (np.abs(got / size - want) / big).astype(float)
    assert err.max() <= 2e-15, err.max()
