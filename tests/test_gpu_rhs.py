"""The push's right-hand side on integer mantissas, at the ends of its ranges:
against an extended-precision step, under powers of two that cancel, with
arguments it hands to the FP64 form, and on nodes its index estimate misses."""
import numpy as np
import pytest

from paper_2602_07452_gb300 import inputs as I
from helpers import cuda_or_skip, dev, fpic, make_particles
from test_gpu_gather import _interp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
L = np.longdouble


def _rhs(a, y, q, D, B):
    r, th, _, ur, ut, up = y
    s, c = np.sin(th), np.cos(th)
    P = r * r + a * a * c * c
    xi = 1 + 2 * r / P
    al = 1 / np.sqrt(xi)
    U = [a / P * (a * s * s * ur + up) + ur / xi, ut / P, a / P * ur + up / (P * s * s)]
    G = np.sqrt(1 + ur * U[0] + ut * U[1] + up * U[2])
    f = [al * U[0] / G - 1 + 1 / xi, al * U[1] / G, al * U[2] / G]
    for i in range(2):
        dP = -2 * a * a * s * c if i else 2 * r
        dxi = -2 * r * dP / P**2 + (0 if i else 2 / P)
        das = 2 * a * a * s * c if i else 0
        quad = (ur**2 * (das / P - a * a * s * s * dP / P**2 - dxi / xi**2) - (2 * ur * up * a + ut**2) * dP / P**2
                + up**2 * (-dP / (P * s) ** 2 - (2 * c / (P * s**3) if i else 0)))
        f.append(G * al * dxi / xi / 2 + ur * dxi / xi**2 - al / G * quad / 2)
    f.append(0 * r)
    k, ks, rp = q * al, q * al * P * np.sqrt(xi) * s / G, -a * xi * s * s
    pp = s * s * (P + a * a * xi * s * s)
    f[3] = f[3] + k * (xi * D[0] + rp * D[2]) + ks * (U[1] * B[2] - U[2] * B[1])
    f[4] = f[4] + k * P * D[1] + ks * (U[2] * B[0] - U[0] * B[2])
    f[5] = f[5] + k * (rp * D[0] + pp * D[2]) + ks * (U[0] * B[1] - U[1] * B[0])
    return f


def _push(z, qm, a, D, B, dt, scale=1.0):
    F = fpic()
    g = I.log_grid(24, 24, 1.9, 30.0)
    ctx = F.fpic_init_metric(1.0, a)
    F.fpic_set_grid(ctx, g)
    n = len(z)
    p = make_particles(z, qm / scale, H0=np.ones(n), D0=np.ones(n), Hn=np.ones(n))
    F.fpic_push(ctx, p, [dev(np.full(g.size, v * scale)) for v in (*D, *B)], F.push_params(dt, scheme=F.FPIC_RK4))
    return np.stack([x.cpu().numpy() for x in (p.r, p.th, p.ph, p.ur, p.uth, p.uph)]), p.alive.cpu().numpy()


def _state(n, size, seed):
    rng = np.random.default_rng(seed)
    z = np.zeros((n, 6))
    z[:, 0] = np.exp(rng.uniform(np.log(2.1), np.log(28.0), n))
    z[:, 1] = rng.uniform(0.1, np.pi - 0.1, n)
    z[:, 3:] = rng.normal(size=(n, 3)) * size
    return z, rng.normal(size=n)


@pytest.mark.parametrize("size", [0.0, 1e-200, 1e-9, 1.0, 1e6])
@pytest.mark.parametrize("a", [0.0, 0.95])
def test_step_against_extended_precision(a, size):
    """Per component: the result's rounding, the four slopes' (each the sum of
    at most a dozen terms, correct to 2^-52 of the largest) and the midpoints'
    roundings times dt and a Jacobian of order ten: 3e-15 of |z| plus dt times
    the slopes' terms."""
    cuda_or_skip()
    D, B, dt = (0.3, -0.2, 0.1), (0.4, 0.1, -0.25), 0.01
    z, qm = _state(4000, size, 5)
    got, _ = _push(z, qm, a, D, B, dt)
    z0, q = [x.astype(L) for x in z.T], qm.astype(L)
    add = lambda h, k: [x + h * y for x, y in zip(z0, k)]
    dt = L(dt)
    k1 = _rhs(L(a), z0, q, D, B)
    k2 = _rhs(L(a), add(dt / 2, k1), q, D, B)
    k3 = _rhs(L(a), add(dt / 2, k2), q, D, B)
    k4 = _rhs(L(a), add(dt, k3), q, D, B)
    term = 1.0 + np.abs(z[:, 3:]).max(1) * (1 + 1 / np.sin(z[:, 1]) ** 3) + np.abs(qm) * z[:, 0] ** 3
    for i in range(6):
        want = z0[i] + dt / 6 * (k1[i] + 2 * k2[i] + 2 * k3[i] + k4[i])
        tol = 3e-15 * (np.abs(z[:, i]) + float(dt) * term)
        assert (np.abs(got[i] - want) <= tol).all(), (i, float((np.abs(got[i] - want) / tol).max()))


@pytest.mark.parametrize("k", [-900, -300, -40, 40, 300, 900])
def test_field_and_charge_scale_cancel_exactly(k):
    """Fields times 2^k and charges over 2^k: the same bits, at any exponent."""
    cuda_or_skip()
    z, qm = _state(3000, 1.0, 6)
    D, B = (0.3, -0.2, 0.1), (0.4, 0.1, -0.25)
    one, _ = _push(z, qm, 0.9, D, B, 0.01)
    assert np.array_equal(one, _push(z, qm, 0.9, D, B, 0.01, 2.0**k)[0])


def test_arguments_without_a_mantissa():
    """NaN and infinite states leave the domain as before, their neighbours
    in the warp step on; a polar axis th = 0 gives what FP64 gives (no number),
    zero momenta and fields exactly zero forces."""
    cuda_or_skip()
    z, qm = _state(256, 0.0, 7)
    ref, _ = _push(z, qm, 0.5, (0, 0, 0), (0, 0, 0), 1e-3)
    assert np.array_equal(ref[5], z[:, 5]) and (ref[2][np.abs(ref[4]) == 0] != np.inf).all()
    bad = z.copy()
    bad[3, 0], bad[40, 0], bad[70, 3], bad[90, 1], bad[130, 5] = np.nan, np.inf, np.nan, np.nan, np.inf
    got, alive = _push(bad, qm, 0.5, (0, 0, 0), (0, 0, 0), 1e-3)
    hit = np.zeros(256, bool)
    hit[[3, 40, 70, 90, 130]] = True
    assert np.array_equal(got[:, ~hit], ref[:, ~hit]) and alive[~hit].all() and not alive[[3, 40]].any()
    assert not np.isfinite(got[3, 70]) and not np.isfinite(got[1, 90]) and not np.isfinite(got[5, 130])


def test_gather_on_nodes_the_estimate_misses():
    """Node lists clustered so that the estimate in ln r and th is many cells
    off: the same gathered force as on even ones (tolerance as in
    test_gpu_gather: 1e-13 and the drift over the step)."""
    cuda_or_skip()
    F = fpic()
    g = I.log_grid(60, 48, 1.9, 30.0)
    t = np.linspace(0.0, 1.0, g.Nth + 1)
    g.tn = g.tn[0] + (g.tn[-1] - g.tn[0]) * (0.2 * t + 0.8 * t**3)
    g.th = 0.5 * (g.tn[:-1] + g.tn[1:])
    g.rn = 1.9 + 28.1 * np.linspace(0.0, 1.0, g.Nr + 1) ** 1.5
    g.rh = 0.5 * (g.rn[:-1] + g.rn[1:])
    ctx = F.fpic_init_metric(1.0, 0.0)
    F.fpic_set_grid(ctx, g)
    rng = np.random.default_rng(9)
    f = [np.zeros(g.size) for _ in range(6)]
    f[2] = rng.normal(size=g.size)
    n, dt = 3000, 1e-9
    r = np.exp(rng.uniform(np.log(2.05), np.log(29.5), n))
    th = rng.uniform(0.02, np.pi - 0.02, n)
    z = np.zeros((n, 6))
    z[:, 0], z[:, 1] = r, th
    p = make_particles(z, np.ones(n), H0=np.ones(n), D0=np.ones(n), Hn=np.ones(n))
    F.fpic_push(ctx, p, [dev(x) for x in f], F.push_params(dt, scheme=F.FPIC_RK4))
    size = (r * np.sin(th)) ** 2 / np.sqrt(1.0 + 2.0 / r)
    err = np.abs(p.uph.cpu().numpy() / dt / size - _interp(g, f[2], 2, r, th)) / np.abs(f[2]).max()
    i = np.clip(np.searchsorted(g.rn, r, side="right") - 1, 0, g.Nr - 1)
    drift = 4.0 * dt / (g.rn[i + 1] - g.rn[i])
    assert (err <= 1e-13 + drift).all(), err.max()
