"""Performance cases: the work a user of this framework has it do, each through its public entry points.

The listed cases are the workloads of this repository's benchmark and tests (the hybrid push of charged particles in
the Wald field, neutral geodesics, batched runs, host-resident particles, the deposits, the field update, divergence
cleaning, whole GRPIC steps, the network's training step) at their own sizes; `draw` spreads the same kinds of work
over sizes from a few hundred to a few million particles and grids from 24 to 1024 cells a side, odd ones among them.

`exact` restates each path in plain 64-bit torch from the equations, without the framework's code.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2602_07452_gb300 import fpic as F
from paper_2602_07452_gb300.grpic import GRPIC

DEV = "cuda"
f64 = torch.float64
QM = 100.0              # |q/m| of the pair plasma
HYB1_THR = 3.5e-6       # Hyb1's energy-rate threshold
LOSS_W = (1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 0.0, 0.1, 0.0)


def listed():
    return [
        # test-particle geodesics of a few thousand particles, one call per step: launches and latency
        dict(name="geodesics_4096", kind="push", scheme="hyb2", neutral=True, n=4096, a=0.9, dt=0.01),
        # the flagship: charged test particles in a fixed Wald field, hybrid RK4 / implicit midpoint
        dict(name="wald_hyb1_2e20", kind="push", scheme="hyb1", neutral=False, n=1 << 20, nr=512, nth=512, a=0.9,
             dt=1e-3),
        # the same workload from pinned host arrays, each step in and out over the link; a ragged size
        dict(name="wald_hyb1_host", kind="push", scheme="hyb1", neutral=False, n=250007, nr=257, nth=200, a=0.9,
             dt=1e-3, host=True),
        # a campaign of independent split-monopole runs advanced in one batch (uneven spins, grids, counts)
        dict(name="monopole_batch", kind="batch", runs=12, n_min=3000, n_max=300000, g_min=128, g_max=512, dt=1e-3),
        # the deposit of a production-like plasma, sort included
        dict(name="deposit_512x16", kind="deposit", nr=512, nth=512, ppc=16, a=0.99),
        # the charge-conserving deposit of the same plasma's moves
        dict(name="deposit_conserving_512x16", kind="deposit_cons", nr=512, nth=512, ppc=16, a=0.99, dt=5e-4),
        # one leapfrog step of the fields with sources and absorbing layer, plasma grid
        dict(name="fdtd_1024", kind="fdtd", nr=1024, nth=1024, a=0.99, full=False),
        # the vacuum magnetosphere on the full-theta domain (periodic), the widest grid in use
        dict(name="fdtd_full_theta", kind="fdtd", nr=4196, nth=1024, a=0.999, full=True),
        # divergence cleaning with the usual 500 sweeps
        dict(name="clean_1024", kind="clean", nr=1024, nth=1024, a=0.99, sweeps=500),
        # a small plasma step (convergence studies, tests): every phase is a short launch
        dict(name="pic_step_96x64x8", kind="pic", nr=96, nth=64, ppc=8, a=0.99, dt=5e-4, conserving=False),
        # the production plasma step: 32 pairs per cell on 1024 x 1024
        dict(name="pic_step_1024x64", kind="pic", nr=1024, nth=1024, ppc=64, a=0.99, dt=5e-4, conserving=False),
        # one training step of the learned guess at its usual minibatch
        dict(name="train_8192", kind="train", batch=8192),
    ]


def draw(rng):
    """One more case of the same kinds; sizes log-uniform, odd ones among them."""
    lg = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    a = round(rng.uniform(0.1, 0.999), 4)
    kind = rng.choice(["push", "push", "push", "batch", "deposit", "deposit", "deposit_cons", "fdtd", "fdtd", "clean",
                       "pic", "pic", "train"])
    if kind == "push":
        scheme = rng.choice(["rk4", "hyb1", "imr"])
        neutral = rng.random() < 0.25
        c = dict(kind=kind, scheme="hyb2" if neutral and scheme != "rk4" else scheme, neutral=neutral,
                 n=lg(300, 3000000), a=a, dt=0.01 if neutral else 1e-3)
        if not neutral:
            c.update(nr=lg(48, 1024), nth=lg(48, 1024))
            if rng.random() < 0.2:
                c["host"], c["n"] = True, min(c["n"], 1000000)
        return c
    if kind == "batch":
        g = lg(64, 256)
        return dict(kind=kind, runs=rng.randint(2, 16), n_min=lg(300, 3000), n_max=lg(3000, 500000), g_min=g,
                    g_max=g + lg(8, 300), dt=1e-3)
    if kind in ("deposit", "deposit_cons", "pic"):
        nr, nth = lg(24, 700), lg(24, 700)
        ppc = 2 * max(1, min(lg(1, 32), 4000000 // (nr * nth)))
        c = dict(kind=kind, nr=nr, nth=nth, ppc=ppc, a=a)
        if kind != "deposit":
            c["dt"] = 5e-4
        if kind == "pic":
            c["conserving"] = rng.random() < 0.3
        return c
    if kind == "fdtd":
        full = rng.random() < 0.4
        return dict(kind=kind, nr=lg(24, 1500), nth=2 * lg(12, 600) if full else lg(24, 1200), a=a, full=full)
    if kind == "clean":
        return dict(kind=kind, nr=lg(24, 1024), nth=lg(24, 1024), a=a, sweeps=rng.randint(20, 500))
    return dict(kind=kind, batch=1 << rng.randint(8, 16))


# ---------------------------------------------------------------------------------------------------------------------
# inputs: plain torch / numpy
# ---------------------------------------------------------------------------------------------------------------------

def horizon(a):
    return 1.0 + math.sqrt(1.0 - a * a)


def make_grid(nr, nth, r_min, r_max, full=False):
    """Node tables uniform in ln r and th (full: one period of th with both poles between a node and a half node)."""
    lr = np.linspace(math.log(r_min), math.log(r_max), nr + 1)
    if full:
        dth = 2.0 * math.pi / nth
        tn = 0.25 * dth + dth * np.arange(nth + 1)
    else:
        dth = math.pi / (nth + 1)
        tn = np.linspace(0.5 * dth, math.pi - 0.5 * dth, nth + 1)
    th = tn[:-1] + 0.5 * dth if full else 0.5 * (tn[:-1] + tn[1:])
    return SimpleNamespace(Nr=nr, Nth=nth, rn=np.exp(lr), rh=np.exp(0.5 * (lr[:-1] + lr[1:])), tn=tn, th=th,
                           ld=nth + 1, size=(nr + 1) * (nth + 1), full_theta=full)


def gen_of(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def uniform(g, n, lo, hi):
    return torch.rand(n, generator=g, dtype=f64, device=DEV) * (hi - lo) + lo


def metric(a, r, s, c):
    """Kerr-Schild (M = 1): rho^2, xi, alpha, beta^r, g^rr, g^rph, g^thth, g^phph, g_rr, g_rph, g_phph, sqrt(gamma)."""
    P = r * r + a * a * c * c
    xi = 1.0 + 2.0 * r / P
    al = xi ** -0.5
    return SimpleNamespace(P=P, xi=xi, al=al, be=2.0 * r / (P * xi), urr=a * a * s * s / P + 1.0 / xi, urp=a / P,
                           utt=1.0 / P, upp=1.0 / (P * s * s), rr=xi, rp=-a * xi * s * s, tt=P,
                           pp=s * s * (P + a * a * xi * s * s), sg=P * xi.sqrt() * s if torch.is_tensor(xi) else None)


def raise_u(m, u):
    return m.urr * u[0] + m.urp * u[2], m.utt * u[1], m.urp * u[0] + m.upp * u[2]


def gamma_of(m, u):
    U = raise_u(m, u)
    return (1.0 + u[0] * U[0] + u[1] * U[1] + u[2] * U[2]).sqrt()


def h_parts(a, z, qm, B0):
    """alpha Gamma - beta u_r and (q/m) A_0 of the Wald potential of strength B0."""
    s, c = z[1].sin(), z[1].cos()
    m = metric(a, z[0], s, c)
    kin = m.al * gamma_of(m, z[3:]) - m.be * z[3]
    pot = qm * (B0 * a) * z[0] * (1.0 + c * c) / m.P
    return kin, pot


def juttner(g, n, theta):
    """Isotropic momenta with |u| from the Maxwell-Juttner law of temperature theta."""
    u = np.linspace(0.0, 40.0 * theta + 8.0 * math.sqrt(theta), 1 << 14)
    pdf = u * u * np.exp(-(np.sqrt(1.0 + u * u) - 1.0) / theta)
    cdf = np.concatenate([[0.0], np.cumsum(0.5 * (pdf[1:] + pdf[:-1]))])
    ut, ct = torch.as_tensor(u, device=DEV), torch.as_tensor(cdf / cdf[-1], device=DEV)
    x = uniform(g, n, 0.0, 1.0)
    k = torch.searchsorted(ct, x, right=True).clamp_(1, len(u) - 1)
    mag = ut[k - 1] + (x - ct[k - 1]) / (ct[k] - ct[k - 1]).clamp_min(1e-300) * (ut[k] - ut[k - 1])
    cz, ph = uniform(g, n, -1.0, 1.0), uniform(g, n, 0.0, 2.0 * math.pi)
    sz = (1.0 - cz * cz).sqrt()
    return mag * sz * ph.cos(), mag * sz * ph.sin(), mag * cz


def momenta(a, r, th, uhat):
    """Covariant momenta of FIDO-frame ones (gamma_ij = L L^T)."""
    m = metric(a, r, th.sin(), th.cos())
    l11, l22 = m.rr.sqrt(), m.tt.sqrt()
    l31 = m.rp / l11
    return l11 * uhat[0], l22 * uhat[1], l31 * uhat[0] + (m.pp - l31 * l31).sqrt() * uhat[2]


def species(n):
    return torch.where(torch.arange(n, device=DEV) % 2 == 0, -QM, QM).to(f64)


AXIS = 0.02     # the particles start outside a narrow cone around the axis, where these steps do not resolve the motion


def thermal(g, n, a, grid, theta):
    """Thermal pairs, uniform in ln r and th over the grid."""
    r = uniform(g, n, math.log(1.02 * horizon(a)), math.log(0.98 * grid.rn[-1])).exp_()
    th = uniform(g, n, max(AXIS, grid.tn[0]), min(math.pi - AXIS, grid.tn[-1]))
    ph = uniform(g, n, 0.0, 2.0 * math.pi)
    return [r, th, ph, *momenta(a, r, th, juttner(g, n, theta))], species(n)


def orbits(g, n, a):
    """Neutral particles on near-Keplerian bound orbits."""
    r = uniform(g, n, 8.0, 20.0)
    th = uniform(g, n, 0.6, math.pi - 0.6)
    L = r.sqrt() * uniform(g, n, 0.98, 1.12)
    return [r, th, uniform(g, n, 0.0, 2.0 * math.pi), uniform(g, n, -0.02, 0.02), 0.3 * L * uniform(g, n, -1.0, 1.0),
            L * th.sin()], torch.zeros(n, dtype=f64, device=DEV)


def plasma(g, a, grid, ppc, theta=0.5):
    """ppc thermal particles in every cell outside the horizon and the cone around the axis, cell by cell."""
    lo = 1.02 * horizon(a)
    i = torch.as_tensor(np.nonzero(grid.rn[1:] > lo)[0], device=DEV)
    j = torch.as_tensor(np.nonzero((grid.tn[:-1] > AXIS) & (grid.tn[1:] < math.pi - AXIS))[0], device=DEV)
    ii = i.repeat_interleave(len(j) * ppc)
    jj = j.repeat_interleave(ppc).repeat(len(i))
    n = ii.numel()
    lr, tn = torch.as_tensor(np.log(grid.rn), device=DEV), torch.as_tensor(grid.tn, device=DEV)
    x = uniform(g, n, 0.0, 1.0)
    r = (lr[ii] + x * (lr[ii + 1] - lr[ii])).exp_().clamp_min_(lo)
    x = uniform(g, n, 0.0, 1.0)
    th = tn[jj] + x * (tn[jj + 1] - tn[jj])
    del ii, jj, x
    ph = uniform(g, n, 0.0, 2.0 * math.pi)
    return [r, th, ph, *momenta(a, r, th, juttner(g, n, theta))], species(n)


def wald_at(a, r, s, c):
    """The Wald field of strength 1 at (r, th): D^i, B^i."""
    m = metric(a, r, s, c)
    P, a2, k = m.P, a * a, 1.0 + c * c
    q = a2 * k - P
    dpt = s * c * (r * r + a2 - 2.0 * a2 * r * k / P - 2.0 * a2 * r * s * s * q / P ** 2)
    dpr = 0.5 * s * s * (2.0 * r - 2.0 * a2 * k * (P - 2.0 * r * r) / P ** 2)
    B = dpt / m.sg, -dpr / m.sg, -a * s * c * (-1.0 + 2.0 * r * q / P ** 2) / m.sg
    Er, Et = a * k * (P - 2.0 * r * r) / P ** 2, 2.0 * a * r * s * c * q / P ** 2
    dr, dt, dp = Er / m.al, (Et + m.sg * m.be * B[2]) / m.al, -m.sg * m.be * B[1] / m.al
    return (m.urr * dr + m.urp * dp, m.utt * dt, m.urp * dr + m.upp * dp), B


# staggering (r half, th half) of D^r, D^th, D^ph, B^r, B^th, B^ph
STAG = ((1, 0), (0, 1), (0, 0), (0, 1), (1, 0), (1, 1))


def points(grid, ro, to):
    r = torch.as_tensor(grid.rh if ro else grid.rn, device=DEV)[:, None]
    th = torch.as_tensor(grid.th if to else grid.tn, device=DEV)[None, :]
    return r, th


def wald_fields(a, grid):
    out = []
    for k, (ro, to) in enumerate(STAG):
        r, th = points(grid, ro, to)
        D, B = wald_at(a, r, th.sin(), th.cos())
        f = torch.zeros(grid.Nr + 1, grid.ld, dtype=f64, device=DEV)
        f[:r.shape[0], :th.shape[1]] = D[k] if k < 3 else B[k - 3]
        if grid.full_theta:
            f[:, grid.Nth] = f[:, 0]
        out.append(f.reshape(-1))
    return out


def monopole_fields(a, grid):
    """The split monopole with a current sheet that these grids and steps resolve."""
    r, th = points(grid, 0, 1)
    x = 5.0 * (th - 0.5 * math.pi)
    zeta, dzeta = (2.0 / math.pi) * x.atan(), (2.0 / math.pi) * 5.0 / (1.0 + x * x)
    m = metric(a, r, th.sin(), th.cos())
    out = [torch.zeros(grid.size, dtype=f64, device=DEV) for _ in range(6)]
    out[3].view(grid.Nr + 1, grid.ld)[:, :grid.Nth] = 4.0 * (dzeta * (1.0 - th.cos()) + zeta * th.sin()) / m.sg
    return out


def push_inputs(case, seed):
    g = gen_of(seed)
    if case["neutral"]:
        z, qm = orbits(g, case["n"], case["a"])
        return z, qm, None, None
    grid = make_grid(case["nr"], case["nth"], 0.9 * horizon(case["a"]), 50.0)
    z, qm = thermal(g, case["n"], case["a"], grid, 0.1)
    return z, qm, grid, wald_fields(case["a"], grid)


def batch_inputs(case, seed):
    k = case["runs"]
    spins = np.linspace(0.5, 0.99, k)
    sides = np.round(np.geomspace(case["g_min"], case["g_max"], k)).astype(int)
    counts = np.round(np.geomspace(case["n_min"], case["n_max"], k)).astype(int)
    g, out = gen_of(seed), []
    for a, side, n in zip(spins, sides, counts):
        grid = make_grid(int(side), int(side), 0.9 * horizon(float(a)), 50.0)
        z, qm = thermal(g, int(n), float(a), grid, 0.1)
        out.append((float(a), grid, z, qm, monopole_fields(float(a), grid)))
    return out


def plasma_inputs(case, seed):
    grid = make_grid(case["nr"], case["nth"], 0.9 * horizon(case["a"]), 50.0)
    z, qm = plasma(gen_of(seed), case["a"], grid, case["ppc"])
    return grid, z, qm


def moved(case, grid, z):
    """The positions a step later of free-streaming particles (well under a cell)."""
    m = metric(case["a"], z[0], z[1].sin(), z[1].cos())
    U, G = raise_u(m, z[3:]), gamma_of(m, z[3:])
    r = z[0] + case["dt"] * (m.al * U[0] / G - m.be)
    th = (z[1] + case["dt"] * m.al * U[1] / G).clamp(grid.tn[0], grid.tn[-1])
    return [r, th, z[2], *z[3:]]


def field_inputs(case, seed):
    """Leapfrog levels near the Wald field with noise, and sources."""
    a = case["a"]
    grid = make_grid(case["nr"], case["nth"], 0.99 * horizon(a), 20.0, case["full"])
    g, w = gen_of(seed), wald_fields(a, grid)

    def noise(k, amp, base=None):
        ro, to = STAG[k]
        x = torch.zeros(grid.Nr + 1, grid.ld, dtype=f64, device=DEV)
        nr, nt = grid.Nr + 1 - ro, grid.ld - to
        x[:nr, :nt] = amp * torch.randn(nr, nt, generator=g, dtype=f64, device=DEV)
        if base is not None:
            x += base.view_as(x)
        if grid.full_theta:
            x[:, grid.Nth] = x[:, 0]
        return x.reshape(-1)

    fl = {}
    for nm, at in (("D0", 0), ("D1", 0), ("B0", 3), ("B1", 3)):
        fl[nm] = [noise(at + k, 1e-3, w[at + k]) for k in range(3)]
    for nm in ("j0", "j1"):
        fl[nm] = [noise(k, 1e-4) for k in range(3)]
    fl["rho0"], fl["rho1"] = noise(2, 1e-4), noise(2, 1e-4)
    return grid, fl, 0.1 * float(grid.rn[1] - grid.rn[0])


def clean_inputs(case, seed):
    grid = make_grid(case["nr"], case["nth"], 0.9 * horizon(case["a"]), 50.0)
    g, w = gen_of(seed), wald_fields(case["a"], grid)
    r = lambda: 1e-3 * torch.randn(grid.size, generator=g, dtype=f64, device=DEV)
    return grid, [w[k] + r() for k in range(3)], r()


def train_inputs(case, seed):
    g, dims, parts = gen_of(seed), (14, 128, 128, 128, 9), []
    rn = lambda *sh: torch.randn(*sh, generator=g, dtype=torch.float32, device=DEV)
    for i, o in zip(dims[:-1], dims[1:]):
        parts += [rn(o * i) * math.sqrt(2.0 / i), 0.01 * rn(o)]
    B = case["batch"]
    X = rn(B, 16)
    X[:, 14:] = 0.0
    return torch.cat(parts), X, rn(B, 16), (torch.rand(B, generator=g, device=DEV) < 0.3).float()


# ---------------------------------------------------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------------------------------------------------

STATE = ("r", "th", "ph", "ur", "uth", "uph")


def fill(p, a, z, qm, w=1.0, B0=0.0):
    for nm, x in zip(STATE, z):
        getattr(p, nm).copy_(x)
    kin, pot = h_parts(a, z, qm, B0)
    p.qm.copy_(qm)
    p.w.fill_(w)
    p.H0.copy_(kin - pot)
    p.Hn.copy_(kin - pot)
    p.D0.copy_(kin.abs() + pot.abs())
    p.alive.fill_(1)
    return p


def context(a, grid=None):
    ctx = F.fpic_init_metric(1.0, a)
    if grid is not None:
        F.fpic_set_grid(ctx, grid)
    return ctx


def push_prm(case, r_max):
    scheme = dict(rk4=F.FPIC_RK4, imr=F.FPIC_IMR, hyb1=F.FPIC_HYB1, hyb2=F.FPIC_HYB2)[case["scheme"]]
    if case["neutral"]:
        return F.push_params(case["dt"], scheme=scheme, implicit=F.FPIC_HAM, thr=1e-12, r_max=r_max)
    return F.push_params(case["dt"], scheme=scheme, implicit=F.FPIC_IMR, thr=HYB1_THR, r_max=r_max, B0pot=1.0,
                         imr_newton=True, imr_substeps=8, substep_tol=1e-4)


def prepare(case, seed):
    k = case["kind"]
    if k == "push":
        z, qm, grid, fields = push_inputs(case, seed)
        ctx = context(case["a"], grid)
        if grid is not None:
            F.fpic_set_tuning(ctx, F.FPIC_TUNE_STATIC_FIELDS, 1)     # test particles: the field stays as it is
        F.fpic_set_tuning(ctx, F.FPIC_TUNE_REUSE_SLOPE, 1)
        host = bool(case.get("host"))
        p = fill(F.HostParticles(case["n"]) if host else F.Particles.empty(case["n"]), case["a"], z, qm,
                 B0=0.0 if grid is None else 1.0)
        call = F.fpic_push_host if host else F.fpic_push
        prm = push_prm(case, 1e300 if grid is None else float(grid.rn[-1]))
        return dict(do=lambda: call(ctx, p, fields, prm), out=lambda: push_out(p, case["scheme"]))
    if k == "batch":
        runs, off, parts = [], 0, batch_inputs(case, seed)
        p = F.Particles.empty(sum(x[3].numel() for x in parts))
        for a, grid, z, qm, fields in parts:
            n = qm.numel()
            fill(F.Particles(*[getattr(p, f)[off:off + n] for f in p.__dataclass_fields__]), a, z, qm)
            runs.append((context(a, grid), fields, off, off + n, float(grid.rn[-1]), 0.0))
            off += n
        table = F.make_runs(runs)
        prm = F.push_params(case["dt"], scheme=F.FPIC_HYB1, implicit=F.FPIC_IMR, thr=HYB1_THR, imr_newton=True)
        return dict(do=lambda: F.fpic_push_batched(table, p, prm), out=lambda: push_out(p, "hyb1"), keep=runs)
    if k in ("deposit", "deposit_cons"):
        grid, z, qm = plasma_inputs(case, seed)
        ctx = context(case["a"], grid)
        p = fill(F.Particles.empty(qm.numel()), case["a"], z, qm, 1e-6)
        if k == "deposit":
            src = tuple(torch.zeros(grid.size, dtype=f64, device=DEV) for _ in range(4))
            return dict(do=lambda: F.fpic_deposit(ctx, p, grid.size, out=src),
                        out=lambda: dict(src=src, **{nm: getattr(p, nm) for nm in STATE}, cell=p.cell))
        q = fill(F.Particles.empty(qm.numel()), case["a"], moved(case, grid, z), qm, 1e-6)
        src = tuple(torch.zeros(grid.size, dtype=f64, device=DEV) for _ in range(4))
        return dict(do=lambda: F.fpic_deposit_conserving(ctx, p, q, case["dt"], out=src), out=lambda: dict(src=src))
    if k == "fdtd":
        grid, init, dt = field_inputs(case, seed)
        ctx = context(case["a"], grid)
        fl = F.Fields(grid.size)
        for nm, arrs in init.items():
            for dst, x in zip(getattr(fl, nm) if isinstance(arrs, list) else [getattr(fl, nm)],
                              arrs if isinstance(arrs, list) else [arrs]):
                dst.copy_(x)
        r_max = float(grid.rn[-1])
        prm = F.fdtd_params(dt, 1e4, 5.0, 0.9 * r_max, r_max)

        def step():
            F.fpic_fdtd_step(ctx, fl, prm, 1)
            F.fpic_fdtd_step(ctx, fl, prm, 2)
            fl.swap()
        return dict(do=step, out=lambda: dict(B0=fl.B0, B1=fl.B1, D0=fl.D0, D1=fl.D1))
    if k == "clean":
        grid, D, rho = clean_inputs(case, seed)
        ctx = context(case["a"], grid)
        return dict(do=lambda: F.fpic_div_clean(ctx, D, rho, case["sweeps"]), out=lambda: dict(D=D))
    if k == "pic":
        grid, z, qm = plasma_inputs(case, seed)
        ctx = context(case["a"], grid)
        p = fill(F.Particles.empty(qm.numel()), case["a"], z, qm, 1e-6)
        del z, qm
        fl = F.Fields(grid.size)
        for i, w in enumerate(wald_fields(case["a"], grid)):
            for nm in ("D0", "D1") if i < 3 else ("B0", "B1"):
                getattr(fl, nm)[i % 3].copy_(w)
        r_max = float(grid.rn[-1])
        sim = GRPIC(ctx, grid, fl, p, p.n, F.push_params(case["dt"], scheme=F.FPIC_RK4, r_max=r_max),
                    F.fdtd_params(case["dt"], 1e4, 5.0, 0.9 * r_max, r_max), conserving=case["conserving"])
        return dict(do=sim.step, out=lambda: dict(B1=fl.B1, D1=fl.D1, j=fl.j0, rho=fl.rho0, Hn=p.Hn, alive=p.alive,
                                                  cell=p.cell, **{nm: getattr(p, nm) for nm in STATE}), keep=sim)
    P, X, T, S = train_inputs(case, seed)
    net, mom, vel, step = F.MLP(), torch.zeros_like(P), torch.zeros_like(P), [0]
    net.set_params(P)

    def train():
        step[0] += 1
        net.train_step(P, mom, vel, X, T, S, LOSS_W, step[0], lr=2e-3)
    return dict(do=train, out=lambda: dict(P=P, mom=mom, vel=vel))


def push_out(p, scheme):
    """The particles after the push: state, H, domain flag, cell and (hybrids) the scheme taken.  The iteration counts
    are a diagnostic of the implicit solver (a convergence test at rounding level), not a result."""
    out = {nm: getattr(p, nm) for nm in STATE + ("Hn", "alive", "cell")}
    if scheme.startswith("hyb"):
        out["scheme"] = p.scheme
    return out


def run(state):
    state["do"]()
    return state["out"]()


def work(case):
    """Bytes: every input read and every output written once.  Flops: the 64-bit operations of the formulas (an RK4
    step 988, a node share quadrature 1798, a sweep 9 a node), multiplications and additions counted singly."""
    k = case["kind"]
    if k == "push":
        return dict(bytes=180.0 * case["n"], flops=(988.0 if case["scheme"] != "imr" else 800.0) * case["n"])
    if k == "batch":
        n = float(np.round(np.geomspace(case["n_min"], case["n_max"], case["runs"])).sum())
        return dict(bytes=180.0 * n, flops=988.0 * n)
    if k == "train":
        return dict(bytes=case["batch"] * 132.0 + 8.0 * 4 * 36233, flops=case["batch"] * 2.2e5)
    nodes = (case["nr"] + 1.0) * (case["nth"] + 1.0)
    if k == "fdtd":
        # levels and sources in (20 arrays), two levels of B and D out and their half-way values (12), metric tables
        return dict(bytes=nodes * 8 * (20 + 12 + 32), flops=nodes * 250.0)
    if k == "clean":
        return dict(bytes=nodes * 8 * 30, flops=nodes * 9.0 * case["sweeps"])
    n = case["nr"] * case["nth"] * float(case["ppc"])
    if k == "deposit":
        return dict(bytes=n * 160.0 + nodes * 32, flops=n * 1798.0)
    if k == "deposit_cons":
        return dict(bytes=n * 97.0 + nodes * 32, flops=n * 260.0)
    return dict(bytes=n * 260.0 + nodes * 8 * 64, flops=n * (988.0 + (260.0 if case["conserving"] else 1798.0)))


# ---------------------------------------------------------------------------------------------------------------------
# the same in 64 bits, from the equations
# ---------------------------------------------------------------------------------------------------------------------

def locate(X, x):
    """Cell and weight of x on the nodes X, both held at the ends."""
    k = (torch.searchsorted(X, x, right=True) - 1).clamp_(0, X.numel() - 2)
    return k, ((x - X[k]) / (X[k + 1] - X[k])).clamp_(0.0, 1.0)


def nodes_of(grid):
    t = lambda x: torch.as_tensor(x, device=DEV)
    return t(grid.rn), t(grid.rh), t(grid.tn), t(grid.th)


def gather(grid, fields, r, th):
    rn, rh, tn, tt = nodes_of(grid)
    at = {0: locate(rn, r), 1: locate(rh, r)}, {0: locate(tn, th), 1: locate(tt, th)}
    v = []
    for (ro, to), f in zip(STAG, fields):
        (i, x), (j, y) = at[0][ro], at[1][to]
        o = i * grid.ld + j
        lo, hi = f[o] + y * (f[o + 1] - f[o]), f[o + grid.ld] + y * (f[o + grid.ld + 1] - f[o + grid.ld])
        v.append(lo + x * (hi - lo))
    return v[:3], v[3:]


def rhs(a, z, qm, grid, fields):
    r, th, u = z[0], z[1], z[3:]
    s, c = th.sin(), th.cos()
    m = metric(a, r, s, c)
    U, G = raise_u(m, u), gamma_of(m, u)
    dP = 2.0 * r, -2.0 * a * a * s * c
    dxi = 2.0 * (m.P - 2.0 * r * r) / m.P ** 2, 4.0 * r * a * a * s * c / m.P ** 2
    f = [m.al * U[0] / G - m.be, m.al * U[1] / G, m.al * U[2] / G]
    for i in range(2):
        das = 2.0 * a * a * s * c if i else 0.0
        drr = das / m.P - a * a * s * s * dP[i] / m.P ** 2 - dxi[i] / m.xi ** 2
        dpp = -dP[i] / (m.P * s) ** 2 - (2.0 * c / (m.P * s ** 3) if i else 0.0)
        quad = u[0] ** 2 * drr + 2.0 * u[0] * u[2] * (-a * dP[i] / m.P ** 2) + u[1] ** 2 * (-dP[i] / m.P ** 2) \
            + u[2] ** 2 * dpp
        f.append(0.5 * G * m.al * dxi[i] / m.xi + u[0] * dxi[i] / m.xi ** 2 - 0.5 * m.al / G * quad)
    f.append(torch.zeros_like(r))
    if fields is not None:
        D, B = gather(grid, fields, r, th)
        k, ks = qm * m.al, qm * m.al * m.sg / G
        f[3] = f[3] + k * (m.rr * D[0] + m.rp * D[2]) + ks * (U[1] * B[2] - U[2] * B[1])
        f[4] = f[4] + k * m.tt * D[1] + ks * (U[2] * B[0] - U[0] * B[2])
        f[5] = f[5] + k * (m.rp * D[0] + m.pp * D[2]) + ks * (U[0] * B[1] - U[1] * B[0])
    return f


def rk4(a, z, qm, grid, fields, dt):
    add = lambda h, k: [x + h * y for x, y in zip(z, k)]
    k1 = rhs(a, z, qm, grid, fields)
    k2 = rhs(a, add(0.5 * dt, k1), qm, grid, fields)
    k3 = rhs(a, add(0.5 * dt, k2), qm, grid, fields)
    k4 = rhs(a, add(dt, k3), qm, grid, fields)
    return [x + dt / 6.0 * (p + 2.0 * q + 2.0 * r + t) for x, p, q, r, t in zip(z, k1, k2, k3, k4)]


def midpoint(a, z, qm, grid, fields, dt, w):
    """The implicit midpoint step by plain iteration from w."""
    for _ in range(40):
        k = rhs(a, [0.5 * (x + y) for x, y in zip(z, w)], qm, grid, fields)
        w = [x + dt * y for x, y in zip(z, k)]
    return w


def push_exact(a, z, qm, grid, fields, dt, scheme, B0):
    """One step in chunks: the state and H afterwards."""
    outs = []
    for b in range(0, qm.numel(), 1 << 21):
        zc, qc = [x[b:b + (1 << 21)] for x in z], qm[b:b + (1 << 21)]
        w = midpoint(a, zc, qc, grid, fields, dt, zc) if scheme == "imr" else rk4(a, zc, qc, grid, fields, dt)
        kin, pot = h_parts(a, w, qc, B0)
        if scheme == "hyb1":
            k0, p0 = h_parts(a, zc, qc, B0)
            bad = ((kin - pot - k0 + p0).abs() >= HYB1_THR * dt * (k0.abs() + p0.abs())).nonzero()[:, 0]
            zi = midpoint(a, [x[bad] for x in zc], qc[bad], grid, fields, dt, [x[bad] for x in w])
            for x, y in zip(w, zi):
                x[bad] = y
            kin, pot = h_parts(a, w, qc, B0)
        lo, hi = w[1] < 0.0, w[1] > math.pi
        w[1] = torch.where(lo, -w[1], torch.where(hi, 2.0 * math.pi - w[1], w[1]))
        w[2] = torch.where(lo | hi, w[2] + math.pi, w[2])
        w[4] = torch.where(lo | hi, -w[4], w[4])
        outs.append(w + [kin - pot])
    return [torch.cat(x) for x in zip(*outs)]


def trapezoid(a, x0, x1, y0, y1):
    """4 x 4-point trapezoid rule of sqrt(gamma) over [x0, x1] x [y0, y1]."""
    acc = 0.0
    for wl, l in zip((0.5, 1.0, 1.0, 0.5), range(4)):
        th = y0 + l * (y1 - y0) / 3.0
        s, c2 = th.sin(), a * a * th.cos() ** 2
        for wk, k in zip((0.5, 1.0, 1.0, 0.5), range(4)):
            r = x0 + k * (x1 - x0) / 3.0
            P = r * r + c2
            acc = acc + wl * wk * s * (P * (P + 2.0 * r)).sqrt()
    return acc * ((x1 - x0) / 3.0) * ((y1 - y0) / 3.0)


def duals(grid, ro, to):
    """Dual-cell edges (lower, upper) of the sub-grid's nodes in r and th."""
    rn, rh, tn, tt = nodes_of(grid)
    e = lambda n, h: (torch.cat([n[:1], h]), torch.cat([h, n[-1:]]))
    r = (rn[:-1], rn[1:]) if ro else e(rn, rh)
    t = (tn[:-1], tn[1:]) if to else e(tn, tt)
    return r[0][:, None], r[1][:, None], t[0][None], t[1][None]


def deposit_exact(a, grid, z, qm, w):
    """w: the particles' weights (0: removed)."""
    rn, rh, tn, tt = nodes_of(grid)
    acc = [torch.zeros(grid.size, dtype=f64, device=DEV) for _ in range(4)]
    for b in range(0, qm.numel(), 1 << 21):
        zc = [x[b:b + (1 << 21)] for x in z]
        m = metric(a, zc[0], zc[1].sin(), zc[1].cos())
        U, G = raise_u(m, zc[3:]), gamma_of(m, zc[3:])
        Q = w[b:b + (1 << 21)] * qm[b:b + (1 << 21)]
        for to_sum, (ro, to) in (((0, 3), (0, 0)), ((1,), (1, 0)), ((2,), (0, 1))):
            X, Y = (rh if ro else rn), (tt if to else tn)
            x, y = zc[0].clamp(X[0], X[-1]), zc[1].clamp(Y[0], Y[-1])
            i, j = locate(X, x)[0], locate(Y, y)[0]
            V = [trapezoid(a, *(e for e in ((X[i], x), (x, X[i + 1]))[p]), *((Y[j], y), (y, Y[j + 1]))[q])
                 for q in range(2) for p in range(2)]
            tot = V[0] + V[1] + V[2] + V[3]
            for q in range(2):
                for p in range(2):
                    share = V[(1 - p) + 2 * (1 - q)] / tot
                    o = (i + p) * grid.ld + j + q
                    for t in to_sum:
                        acc[t].index_add_(0, o, Q * share if t == 0 else Q * U[(t - 1)] / G * share)
    out = []
    for t, (ro, to) in enumerate(((0, 0), (1, 0), (0, 1), (0, 0))):
        f = torch.zeros(grid.Nr + 1, grid.ld, dtype=f64, device=DEV)
        d = 2.0 * math.pi * trapezoid(a, *duals(grid, ro, to))
        f[:d.shape[0], :d.shape[1]] = acc[t].view(grid.Nr + 1, grid.ld)[:d.shape[0], :d.shape[1]] / d
        out.append(f.reshape(-1))
    return out


def conserving_exact(a, grid, z0, z1, qm, w, dt):
    rn, rh, tn, tt = nodes_of(grid)
    sh = (grid.Nr + 1, grid.ld)
    acc = [torch.zeros(grid.size, dtype=f64, device=DEV) for _ in range(4)]
    i0, f0 = locate(rn, z0[0])
    j0, g0 = locate(tn, z0[1])
    i1, f1 = locate(rn, z1[0])
    j1, g1 = locate(tn, z1[1])
    ib, jb = torch.minimum(i0, i1), torch.minimum(j0, j1)
    ok = ((i0 - i1).abs() <= 1) & ((j0 - j1).abs() <= 1)
    Q = w * qm * ok
    wt = lambda k, base, f: [torch.where(k - base == x, 1.0 - f, torch.where(k - base + 1 == x, f, 0.0))
                             for x in range(3)]
    R0, R1, T0, T1 = wt(i0, ib, f0), wt(i1, ib, f1), wt(j0, jb, g0), wt(j1, jb, g1)
    phd = 0.0
    for z in (z0, z1):
        m = metric(a, z[0], z[1].sin(), z[1].cos())
        phd = phd + 0.5 * m.al * raise_u(m, z[3:])[2] / gamma_of(m, z[3:])

    def put(t, x, y, v):
        i, j = ib + x, jb + y
        acc[t].index_add_(0, (i.clamp_max(grid.Nr) * grid.ld + j.clamp_max(grid.Nth)), v)
    for x in range(3):
        for y in range(3):
            put(0, x, y, Q * R1[x] * T1[y])
            put(3, x, y, Q * phd * 0.5 * (R0[x] * T0[y] + R1[x] * T1[y]))
    for y in range(3):
        s = 0.0
        for x in range(2):
            s = s + (R1[x] - R0[x]) * 0.5 * (T0[y] + T1[y])
            put(1, x, y, -Q * s)
    for x in range(3):
        s = 0.0
        for y in range(2):
            s = s + 0.5 * (R0[x] + R1[x]) * (T1[y] - T0[y])
            put(2, x, y, -Q * s)
    dr = torch.cat([rh, rn[-1:]]) - torch.cat([rn[:1], rh])
    pi = torch.full_like(tt[:1], math.pi)
    dth = torch.cat([tt, pi]) - torch.cat([0.0 * pi, tt])
    out = []
    for t, (ro, to) in enumerate(((0, 0), (1, 0), (0, 1), (0, 0))):
        r, th = points(grid, ro, to)
        d = 2.0 * math.pi * metric(a, r, th.sin(), th.cos()).sg
        d = d * (dt if ro else dr[:, None]) * (dt if to else dth[None])
        f = torch.zeros(sh, dtype=f64, device=DEV)
        f[:d.shape[0], :d.shape[1]] = acc[t].view(sh)[:d.shape[0], :d.shape[1]] / d
        out.append(f.reshape(-1))
    return out


class Leapfrog:
    """The field update from the equations, on whole arrays (Nr + 1, Nth + 1)."""

    def __init__(self, a, grid, dt, conserving=False):
        self.grid, self.dt, self.cons = grid, dt, conserving
        self.N, self.M = grid.Nr, grid.Nth
        self.m = {}
        for ro in (0, 1):
            for to in (0, 1):
                r, th = points(grid, ro, to)
                m = metric(a, r, th.sin(), th.cos())
                m.sg, m.pp, m.rp = (x.expand(r.shape[0], th.shape[1]) for x in (m.sg, m.pp, m.rp))
                self.m[ro, to] = m
        rn, rh, tn, tt = nodes_of(grid)
        r_max, r_abs = float(grid.rn[-1]), 0.9 * float(grid.rn[-1])
        chi = lambda r: torch.exp(-dt * 1e4 * ((r - r_abs) / (r_max - r_abs)).clamp_min(0.0) ** 5.0)[:, None]
        self.dn, self.dh = chi(rn), chi(rh)
        self.drn, self.dtn = (rn[1:] - rn[:-1])[:, None], (tn[1:] - tn[:-1])[None]
        self.drh, self.dth = (rh[1:] - rh[:-1])[:, None], (tt[1:] - tt[:-1])[None]
        if grid.full_theta:
            seam = (tt[:1] + 2.0 * math.pi - tt[-1:])[None]
            self.dth = torch.cat([seam, self.dth], 1)

    def at(self, X, ro, to):
        return X[:self.N + 1 - ro, :self.M + 1 - to]

    def avg(self, X, ro, to):
        """The metric-weighted mean to the other r staggering."""
        v = self.at(X, ro, to) * self.m[ro, to].sg
        if ro:
            v = torch.cat([v[:1], v, v[-1:]])
        return 0.5 * (v[:-1] + v[1:]) / self.m[1 - ro, to].sg

    def put(self, v):
        out = torch.zeros(self.N + 1, self.M + 1, dtype=f64, device=DEV)
        out[:v.shape[0], :v.shape[1]] = v
        if self.grid.full_theta:
            out[:, self.M] = out[:, 0]
        return out

    def E(self, D, B):
        m1, m2, m0 = self.m[1, 0], self.m[0, 1], self.m[0, 0]
        return [self.put(m1.al * (m1.rr * self.at(D[0], 1, 0) + m1.rp * self.avg(D[2], 0, 0))),
                self.put(m2.al * m2.tt * self.at(D[1], 0, 1) - m2.sg * m2.be * self.avg(B[2], 1, 1)),
                self.put(m0.al * (m0.rp * self.avg(D[0], 1, 0) + m0.pp * D[2]) + m0.sg * m0.be * self.avg(B[1], 1, 0))]

    def H(self, D, B):
        m2, m1, m3 = self.m[0, 1], self.m[1, 0], self.m[1, 1]
        return [self.put(m2.al * (m2.rr * self.at(B[0], 0, 1) + m2.rp * self.avg(B[2], 1, 1))),
                self.put(m1.al * m1.tt * self.at(B[1], 1, 0) + m1.sg * m1.be * self.avg(D[2], 0, 0)),
                self.put(m3.al * (m3.rp * self.avg(B[0], 0, 1) + m3.pp * self.at(B[2], 1, 1))
                         - m3.sg * m3.be * self.avg(D[1], 0, 1))]

    def stepB(self, B, E):
        N, M = self.N, self.M
        c0 = (E[2][:, 1:] - E[2][:, :-1]) / self.dtn
        c1 = -(E[2][1:] - E[2][:-1]) / self.drn
        c2 = (E[1][1:, :M] - E[1][:-1, :M]) / self.drn - (E[0][:N, 1:] - E[0][:N, :-1]) / self.dtn
        return [self.put((self.at(B[0], 0, 1) - self.dt * c0 / self.m[0, 1].sg) * self.dn),
                self.put((self.at(B[1], 1, 0) - self.dt * c1 / self.m[1, 0].sg) * self.dh),
                self.put((self.at(B[2], 1, 1) - self.dt * c2 / self.m[1, 1].sg) * self.dh)]

    def J(self, j, rho):
        if self.cons:
            return [self.at(j[0], 1, 0), self.at(j[1], 0, 1), j[2]]
        m1 = self.m[1, 0]
        return [m1.al * self.at(j[0], 1, 0) - self.avg(rho, 0, 0) * m1.be, self.m[0, 1].al * self.at(j[1], 0, 1),
                self.m[0, 0].al * j[2]]

    def stepD(self, D, H, J, old):
        """Interior update, then the boundaries; `old`: the arrays written into (their padding stays)."""
        N, M, full, dt, k = self.N, self.M, self.grid.full_theta, self.dt, 4.0 * math.pi
        lo = 0 if full else 1
        cols = slice(lo, M)
        back = lambda X: (X[:, :M] - torch.cat([X[:, M - 1:M], X[:, :M - 1]], 1)) if full else X[:, 1:M] - X[:, :M - 1]
        out = [x.clone() for x in old]
        out[0][:N, cols] = (D[0][:N, cols] + dt * (back(H[2])[:N] / self.dth / self.m[1, 0].sg[:, cols]
                                                   - k * J[0][:, cols])) * self.dh
        out[1][1:N, :M] = (D[1][1:N, :M] + dt * (-(H[2][1:N, :M] - H[2][:N - 1, :M]) / self.drh
                                                 / self.m[0, 1].sg[1:N] - k * J[1][1:N])) * self.dn[1:N]
        c2 = (H[1][1:N, cols] - H[1][:N - 1, cols]) / self.drh - back(H[0])[1:N] / self.dth
        out[2][1:N, cols] = (D[2][1:N, cols] + dt * (c2 / self.m[0, 0].sg[1:N, cols] - k * J[2][1:N, cols])) \
            * self.dn[1:N]
        if full:
            for x in out:
                x[:, M] = x[:, 0]
        else:
            out[0][:N, 0], out[0][:N, M] = out[0][:N, 1].clone(), out[0][:N, M - 1].clone()
        w1 = slice(0, M + 1) if full else slice(0, M)
        w2 = slice(0, M + 1) if full else slice(1, M)
        out[1][0, w1], out[1][N, w1] = out[1][1, w1].clone(), out[1][N - 1, w1].clone()
        out[2][0, w2], out[2][N, w2] = out[2][1, w2].clone(), out[2][N - 1, w2].clone()
        if not full:
            out[2][:, 0] = out[2][:, M] = 0.0
        return out

    def first(self, f):
        """Sub-steps 1-4: B^{n+3/2} and B^{n+2}."""
        mean = lambda p, q: [0.5 * (x + y) for x, y in zip(f[p], f[q])]
        f["Bh"] = self.stepB(mean("B0", "B1"), self.E(mean("D0", "D1"), f["B1"]))
        f["B2"] = self.stepB(f["B1"], self.E(f["D1"], f["Bh"]))

    def second(self, f):
        """Sub-steps 7-10: D^{n+5/2}; then the levels move on."""
        mean = lambda p, q: [0.5 * (x + y) for x, y in zip(f[p], f[q])]
        J0, J1 = self.J(f["j0"], f["rho0"]), self.J(f["j1"], f["rho1"])
        zero = [torch.zeros_like(x) for x in f["D0"]]
        Dw = self.stepD(mean("D0", "D1"), self.H(f["D1"], f["Bh"]), [0.5 * (x + y) for x, y in zip(J0, J1)], zero)
        D2 = self.stepD(f["D1"], self.H(Dw, f["B2"]), J1, f["D0"])
        return dict(B0=f["B1"], B1=f["B2"], D0=f["D1"], D1=D2)


def clean_exact(a, grid, D, rho, sweeps):
    rn, rh, tn, tt = nodes_of(grid)
    N, M = grid.Nr, grid.Nth
    m = {k: metric(a, *((lambda r, th: (r, th.sin(), th.cos()))(*points(grid, *k)))) for k in ((0, 0), (1, 0), (0, 1))}
    D = [x.view(N + 1, M + 1).clone() for x in D]
    pi = torch.full_like(tt[:1], math.pi)
    dth = (torch.cat([tt, pi]) - torch.cat([0.0 * pi, tt]))[None]
    dr = (rh[1:] - rh[:-1])[:, None]
    fr = m[1, 0].sg * D[0][:N]
    ft = torch.nn.functional.pad(m[0, 1].sg * D[1][:, :M], (1, 1))
    b = (fr[1:] - fr[:-1]) / dr + ((ft[:, 1:] - ft[:, :-1]) / dth)[1:N] \
        - (4.0 * math.pi * m[0, 0].sg * rho.view(N + 1, M + 1))[1:N]
    inv = lambda g: g.pp / (g.rr * g.pp - g.rp ** 2)
    cr = m[1, 0].sg * inv(m[1, 0]) / (rn[1:] - rn[:-1])[:, None]
    ct = torch.nn.functional.pad(m[0, 1].sg / (m[0, 1].tt * (tn[1:] - tn[:-1])[None]), (1, 1))[1:N]
    r1, r0, t1, t0 = cr[1:] / dr, cr[:-1] / dr, ct[:, 1:] / dth, ct[:, :-1] / dth
    tot = r1 + r0 + t1 + t0
    r1, r0, t1, t0, b = r1 / tot, r0 / tot, t1 / tot, t0 / tot, b / tot
    phi = torch.zeros(N + 1, M + 1, dtype=f64, device=DEV)
    for _ in range(sweeps):
        new = r1 * phi[2:] + r0 * phi[:-2] - b
        new[:, :M] += t1[:, :M] * phi[1:N, 1:]
        new[:, 1:] += t0[:, 1:] * phi[1:N, :M]
        phi[1:N] = new
    up = (phi[1:] - phi[:-1]) / (rn[1:] - rn[:-1])[:, None]
    mean = torch.cat([up[:1], 0.5 * (up[:-1] + up[1:]), up[-1:]])
    g = m[0, 0]
    D[0][:N] -= inv(m[1, 0]) * up
    D[1][:, :M] -= (phi[:, 1:] - phi[:, :-1]) / (m[0, 1].tt * (tn[1:] - tn[:-1])[None])
    D[2] -= -g.rp / (g.rr * g.pp - g.rp ** 2) * mean
    return dict(D=[x.reshape(-1) for x in D])


def pic_exact(case, seed):
    a, dt, cons = case["a"], case["dt"], case["conserving"]
    grid, z, qm = plasma_inputs(case, seed)
    v = lambda x: x.view(grid.Nr + 1, grid.ld)
    w = [v(x) for x in wald_fields(a, grid)]
    zero = lambda: torch.zeros(grid.Nr + 1, grid.ld, dtype=f64, device=DEV)
    f = dict(D0=w[:3], D1=w[:3], B0=w[3:], B1=w[3:], j0=[zero() for _ in range(3)], rho0=zero())
    lf = Leapfrog(a, grid, dt, cons)
    lf.first(f)
    *zn, Hn = push_exact(a, z, qm, grid, [x.reshape(-1) for x in f["D1"] + f["Bh"]], dt, "rk4", 0.0)
    gone = (zn[0] < horizon(a)) | (zn[0] > float(grid.rn[-1]))
    src = conserving_exact(a, grid, z, zn, qm, 1e-6, dt) if cons else \
        deposit_exact(a, grid, zn, qm, torch.where(gone, 0.0, torch.full_like(qm, 1e-6)))
    f["rho1"], f["j1"] = v(src[0]), [v(x) for x in src[1:]]
    out = lf.second(f)
    if not cons:                    # the deposit leaves the particles sorted by cell, removed ones last
        rn, _, tn, _ = nodes_of(grid)
        cell = locate(rn, zn[0])[0] * grid.Nth + locate(tn, zn[1])[0]
        order = torch.sort(torch.where(gone, grid.Nr * grid.Nth, cell), stable=True)[1]
        zn, Hn = [x[order] for x in zn], Hn[order]
    flat = lambda xs: [x.reshape(-1) for x in xs]
    return dict(B1=flat(out["B1"]), D1=flat(out["D1"]), j=src[1:], rho=src[0], Hn=Hn, alive=None, cell=None,
                **dict(zip(STATE, zn)))


def train_exact(case, seed):
    P, X, T, S = (x.double() for x in train_inputs(case, seed))
    P.requires_grad_(True)
    h, o = X[:, :14], 0
    for k, (i, n) in enumerate(((14, 128), (128, 128), (128, 128), (128, 9))):
        W, o = P[o:o + n * i].view(n, i), o + n * i
        h, o = h @ W.T + P[o:o + n], o + n
        h = h.relu() if k < 3 else h
    lw = torch.tensor(LOSS_W, dtype=f64, device=DEV)
    loss = ((h - T[:, :9]) ** 2 @ lw + torch.nn.functional.softplus(h[:, 6]) - S * h[:, 6]).mean()
    g, = torch.autograd.grad(loss, P)
    mom, vel = 0.1 * g, 0.001 * g * g
    return dict(P=(P - 2e-3 * (mom / 0.1) / ((vel / 0.001).sqrt() + 1e-8)).detach(), mom=mom, vel=vel)


def exact(case, seed):
    k = case["kind"]
    if k == "push":
        z, qm, grid, fields = push_inputs(case, seed)
        dev = "cpu" if case.get("host") else DEV
        scheme = "rk4" if case["scheme"] == "hyb2" else case["scheme"]      # neutral hybrids keep their RK4 steps
        out = push_exact(case["a"], z, qm, grid, fields, case["dt"], scheme, 0.0 if grid is None else 1.0)
        return dict(zip(STATE + ("Hn",), (x.to(dev) for x in out)))
    if k == "batch":
        outs = [push_exact(a, z, qm, grid, fields, case["dt"], "hyb1", 0.0)
                for a, grid, z, qm, fields in batch_inputs(case, seed)]
        return dict(zip(STATE + ("Hn",), (torch.cat(x) for x in zip(*outs))))
    if k == "deposit":
        grid, z, qm = plasma_inputs(case, seed)
        return dict(src=deposit_exact(case["a"], grid, z, qm, torch.full_like(qm, 1e-6)))
    if k == "deposit_cons":
        grid, z, qm = plasma_inputs(case, seed)
        return dict(src=conserving_exact(case["a"], grid, z, moved(case, grid, z), qm, 1e-6, case["dt"]))
    if k == "fdtd":
        grid, fl, dt = field_inputs(case, seed)
        v = lambda x: [y.view(grid.Nr + 1, grid.ld) for y in x] if isinstance(x, list) else x.view(grid.Nr + 1, grid.ld)
        f = {nm: v(x) for nm, x in fl.items()}
        lf = Leapfrog(case["a"], grid, dt)
        lf.first(f)
        return {nm: [x.reshape(-1) for x in xs] for nm, xs in lf.second(f).items()}
    if k == "clean":
        grid, D, rho = clean_inputs(case, seed)
        return clean_exact(case["a"], grid, D, rho, case["sweeps"])
    if k == "pic":
        return pic_exact(case, seed)
    return train_exact(case, seed)
