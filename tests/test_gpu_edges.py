"""Grids at the edges of the kernels' tiles: the fused leapfrog (31 columns a
warp, up to 16 rows), the cleaning sweeps (two rows a warp, 32 columns), and
more runs in a batch than one launch of the interpolation coefficients takes."""
import numpy as np
import pytest

import oracle as O
from oracle import pic as P
from paper_2602_07452_gb300 import inputs as I
from helpers import cuda_or_skip, dev, fpic, make_particles
from test_gpu_pic import FAMILY, STAG, _fill_random, valid

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nr,nth", [(2, 2), (3, 2), (2, 30), (5, 31), (4, 32), (16, 61), (17, 62), (33, 93)])
def test_leapfrog_on_ragged_grids(nr, nth):
    """Both stages with the absorbing layer, as test_fdtd_step_matches_oracle: 1e-12 of each array's size."""
    cuda_or_skip()
    F = fpic()
    g = I.log_grid(nr, nth, 1.5, 30.0)
    ctx = F.fpic_init_metric(1.0, 0.9)
    F.fpic_set_grid(ctx, g)
    st, fl = P.FdtdState(g), F.Fields(g.size)
    _fill_random(st, fl, g, 9)
    lay = (5.0, 0.6 * g.rn[-1], g.rn[-1])
    po, pg = P.FdtdParams(1.0, 0.9, 0.003, 1e4, *lay), F.fdtd_params(0.003, 1e4, *lay)
    for stage in (1, 2):
        P.fdtd(po, st, stage)
        F.fpic_fdtd_step(ctx, fl, pg, stage)
        for nm in ("B0", "B1", "D0", "D1", "Bh", "E", "H") + (("Dw",) if stage == 2 else ()):
            for k in range(3):
                m = valid(g, nm, k)
                exp, got = getattr(st, nm)[k][m], getattr(fl, nm)[k].cpu().numpy()[m]
                assert np.abs(got - exp).max(initial=0.0) <= 1e-12 * (np.abs(exp).max(initial=0.0) + 1e-300), (stage, nm, k)


@pytest.mark.parametrize("nr,nth", [(2, 4), (5, 30), (7, 32), (16, 62), (17, 124)])
def test_full_theta_leapfrog_on_ragged_grids(nr, nth):
    """The same in the full-theta domain, as test_full_theta_fdtd_step_matches_oracle: columns 0 and Nth bitwise alike."""
    cuda_or_skip()
    F = fpic()
    g = I.full_theta_grid(nr, nth, 1.5, 30.0)
    ctx = F.fpic_init_metric(1.0, 0.9)
    F.fpic_set_grid(ctx, g)
    st, fl = P.FdtdState(g), F.Fields(g.size)
    rng = np.random.default_rng(19)

    def draw():
        x = rng.normal(size=(g.Nr + 1, g.ld))
        x[:, g.Nth] = x[:, 0]
        return x.ravel()

    for nm in ("B0", "B1", "D0", "D1", "j0", "j1"):
        for k in range(3):
            getattr(st, nm)[k][:] = x = draw()
            getattr(fl, nm)[k].copy_(dev(x))
    for nm in ("rho0", "rho1"):
        setattr(st, nm, draw())
        getattr(fl, nm).copy_(dev(getattr(st, nm)))
    lay = (5.0, 0.6 * g.rn[-1], g.rn[-1])
    po, pg = P.FdtdParams(1.0, 0.9, 0.002, 1e4, *lay, 0, 1), F.fdtd_params(0.002, 1e4, *lay)
    for stage in (1, 2):
        P.fdtd(po, st, stage)
        F.fpic_fdtd_step(ctx, fl, pg, stage)
        for nm in ("B0", "B1", "D0", "D1", "Bh", "E", "H") + (("Dw",) if stage == 2 else ()):
            for k in range(3):
                n = g.Nr + 1 - STAG[FAMILY[nm]][k][0]
                exp = getattr(st, nm)[k].reshape(g.Nr + 1, g.ld)[:n]
                got = getattr(fl, nm)[k].cpu().numpy().reshape(g.Nr + 1, g.ld)[:n]
                assert np.abs(got - exp).max() <= 1e-12 * (np.abs(exp).max() + 1e-300), (stage, nm, k)
                assert np.array_equal(got[:, g.Nth], got[:, 0]), (stage, nm, k)


@pytest.mark.parametrize("nr,nth,n_iter", [(2, 2, 3), (3, 31, 4), (4, 32, 5), (9, 33, 7), (10, 70, 8)])
def test_cleaning_on_ragged_grids(nr, nth, n_iter):
    """As test_div_clean_matches_oracle: 1e-10 of the scale."""
    cuda_or_skip()
    F = fpic()
    g = I.log_grid(nr, nth, 1.5, 30.0)
    ctx = F.fpic_init_metric(1.0, 0.9)
    F.fpic_set_grid(ctx, g)
    rng = np.random.default_rng(31 + nr)
    D, rho = [rng.normal(size=g.size) for _ in range(3)], rng.normal(size=g.size) * 0.1
    Dd = [dev(x) for x in D]
    phi = F.fpic_div_clean(ctx, Dd, dev(rho), n_iter, want_phi=True).cpu().numpy()
    Dc, phio = P.div_clean(1.0, 0.9, g, D, rho, n_iter)
    sc = max(np.abs(x).max() for x in Dc)
    assert all(np.abs(Dd[k].cpu().numpy() - Dc[k]).max() <= 1e-10 * sc for k in range(3))
    assert np.abs(phi - phio).max() <= 1e-10 * (np.abs(phio).max() + 1e-300)


@pytest.mark.parametrize("nruns", [32, 33, 65])
def test_batches_of_more_runs_than_a_coefficient_launch(nruns):
    """Bitwise the runs pushed one by one; grids and fields of all sizes within the batch."""
    cuda_or_skip()
    F = fpic()
    specs, alone, zs, qs, n = [], [], [], [], 40
    for k in range(nruns):
        a, g = 0.5 + 0.4 * k / nruns, I.wald_grid(12 + k % 9, 0.9, r_max=30.0)
        ctx = F.fpic_init_metric(1.0, a)
        F.fpic_set_grid(ctx, g)
        f = [dev(x) for x in O.wald_on_grid(a, 1.0, g)]
        d, q, _ = I.thermal_draws(n, g, 3.0, 28.0, 0.1, seed=k)
        zs.append(O.seed_fido(1.0, a, d))
        qs.append(q)
        specs.append((ctx, f, k * n, (k + 1) * n, float(g.rn[-1]), 0.0))
    one = np.ones(nruns * n)
    p = make_particles(np.concatenate(zs), np.concatenate(qs), one, one, one)
    F.fpic_push_batched(F.make_runs(specs), p, F.push_params(1e-3, scheme=F.FPIC_RK4))
    got = p.state().cpu().numpy()
    for k, (ctx, f, b, e, r_max, _) in enumerate(specs):
        p1 = make_particles(zs[k], qs[k], np.ones(n), np.ones(n), np.ones(n))
        F.fpic_push(ctx, p1, f, F.push_params(1e-3, scheme=F.FPIC_RK4, r_max=r_max))
        assert np.array_equal(got[b:e], p1.state().cpu().numpy()), k
