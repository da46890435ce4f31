"""The push's field gather from paired coefficients: cells that are no ordinary
numbers, and the weights at nodes and ends, against plain FP64 interpolation."""
import numpy as np
import pytest

from paper_2602_07452_gb300 import inputs as I
from helpers import cuda_or_skip, dev, fpic, make_particles

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
STAG = ((1, 0), (0, 1), (0, 0), (0, 1), (1, 0), (1, 1))


def _interp(g, f, k, r, th):
    X, Y = (g.rh if STAG[k][0] else g.rn), (g.th if STAG[k][1] else g.tn)
    i = np.clip(np.searchsorted(X, r, side="right") - 1, 0, len(X) - 2)
    j = np.clip(np.searchsorted(Y, th, side="right") - 1, 0, len(Y) - 2)
    x = np.clip((r - X[i]) / (X[i + 1] - X[i]), 0, 1)
    y = np.clip((th - Y[j]) / (Y[j + 1] - Y[j]), 0, 1)
    f = f.reshape(g.Nr + 1, g.ld)
    lo = f[i, j] + y * (f[i, j + 1] - f[i, j])
    return lo + x * (f[i + 1, j] + y * (f[i + 1, j + 1] - f[i + 1, j]) - lo)


@pytest.mark.parametrize("scale", [1.0, 1e-26, 1e-60, 1e40])
def test_force_of_gathered_fields(scale):
    """A step so short that u_ph changes by dt times the force alone, a = 0,
    D^ph and q/m scaled against each other, particles inside cells, on nodes
    and past both ends: u_ph / (q/m dt) is alpha r^2 sin^2 th D^ph to rounding
    (the gather's 2^-47 of the cell's differences and a few FP64 roundings:
    1e-13 of the field's size), at field sizes inside the paired range and
    outside it, where the cells are gathered in FP64."""
    cuda_or_skip()
    F = fpic()
    g = I.log_grid(40, 33, 1.9, 30.0)
    ctx = F.fpic_init_metric(1.0, 0.0)
    F.fpic_set_grid(ctx, g)
    rng = np.random.default_rng(3)
    f = [np.zeros(g.size) for _ in range(6)]
    f[2] = rng.normal(size=g.size) * scale
    n = 4000
    r = np.exp(rng.uniform(np.log(2.05), np.log(29.5), n))
    th = rng.uniform(0.02, np.pi - 0.02, n)
    r[:20], r[20:40] = g.rn[5:25], g.rh[5:25]
    th[40:60], th[60:80] = g.tn[5:25], g.th[5:25]
    z = np.zeros((n, 6))
    z[:, 0], z[:, 1] = r, th
    dt, qm = 1e-9, 1.0 / scale
    p = make_particles(z, np.full(n, qm), H0=np.ones(n), D0=np.ones(n), Hn=np.ones(n))
    F.fpic_push(ctx, p, [dev(x) for x in f], F.push_params(dt, scheme=F.FPIC_RK4))
    al = 1.0 / np.sqrt(1.0 + 2.0 / r)
    want = qm * al * (r * np.sin(th)) ** 2 * _interp(g, f[2], 2, r, th)
    got = p.uph.cpu().numpy() / dt
    # over the step itself r falls by dt beta^r: 1e-9 of it moves the field by 1e-8 of a cell's difference
    size = qm * al * (r * np.sin(th)) ** 2 * np.abs(f[2]).max()
    err = np.abs(got - want) / size
    drift = 4.0 * dt / (r * np.log(g.rn[1] / g.rn[0]))
    assert (err <= 1e-13 + drift).all(), err.max()


def test_a_cell_with_no_number_stays_one():
    """A field value that is NaN or infinite reaches every particle of the
    cells it belongs to (they leave the domain), and no other."""
    cuda_or_skip()
    F = fpic()
    g = I.log_grid(24, 24, 1.9, 30.0)
    ctx = F.fpic_init_metric(1.0, 0.0)
    F.fpic_set_grid(ctx, g)
    for bad in (np.nan, np.inf):
        f = [np.full(g.size, 0.1) for _ in range(6)]
        f[2].reshape(g.Nr + 1, g.ld)[10, 12] = bad
        ii, jj = np.meshgrid(np.arange(3, 22), np.arange(2, 22), indexing="ij")
        r, th = (0.5 * (g.rn[ii] + g.rn[ii + 1])).ravel(), (0.5 * (g.tn[jj] + g.tn[jj + 1])).ravel()
        z = np.zeros((r.size, 6))
        z[:, 0], z[:, 1] = r, th
        p = make_particles(z, np.ones(r.size), H0=np.ones(r.size), D0=np.ones(r.size), Hn=np.ones(r.size))
        F.fpic_push(ctx, p, [dev(x) for x in f], F.push_params(1e-6, scheme=F.FPIC_RK4))
        hit = ((ii == 9) | (ii == 10)) & ((jj == 11) | (jj == 12))
        fine = np.isfinite(p.uph.cpu().numpy())
        assert np.array_equal(fine, ~hit.ravel())
