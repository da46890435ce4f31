"""The charge-conserving deposit of more particles than its record buffer holds
at a time."""
import pytest

from paper_2602_07452_gb300 import inputs as I
from helpers import cuda_or_skip, fpic

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _set(F, n, r, th, u, qm):
    p = F.Particles.empty(n)
    p.r.copy_(r)
    p.th.copy_(th)
    for d, x in zip((p.ur, p.uth, p.uph), u):
        d.copy_(x)
    p.qm.copy_(qm)
    p.w.fill_(1.0)
    p.alive.fill_(1)
    return p


def test_chunks_add_up():
    """Chunk borders fall anywhere among the sorted moves (inside a cell's, at a
    fraction of the moves across boundaries): the whole set's sums are those of
    its two halves, each in one piece, to the roundings of a node's 2 x 10^4
    additions (2^-53 each, of the sum of the terms' sizes: the deposit of |q|),
    and the same bits when repeated."""
    cuda_or_skip()
    F = fpic()
    a, n = 0.9, 70_000_000
    g = I.log_grid(130, 127, 0.9 * I.horizon(1.0, a), 20.0)
    ctx = F.fpic_init_metric(1.0, a)
    F.fpic_set_grid(ctx, g)
    gen = torch.Generator(device="cuda").manual_seed(n)
    rnd = lambda lo, hi: torch.rand(n, generator=gen, dtype=torch.float64, device="cuda") * (hi - lo) + lo
    r, th = rnd(1.6, 19.0), rnd(0.1, 3.0)
    u = [rnd(-1, 1) for _ in range(3)]
    qm = torch.sign(rnd(-1, 1))
    moved = r * (1 + 1e-3 * rnd(-1, 1)), th + 1e-3 * rnd(-1, 1)

    def deposit(sl, sign=True):
        q = qm[sl] if sign else qm[sl].abs()
        m = q.numel()
        return F.fpic_deposit_conserving(ctx, _set(F, m, r[sl], th[sl], [x[sl] for x in u], q),
                                         _set(F, m, moved[0][sl], moved[1][sl], [x[sl] for x in u], q), 1e-3)

    whole = deposit(slice(0, n))
    assert all(torch.equal(x, y) for x, y in zip(whole, deposit(slice(0, n))))
    h = n // 2
    half, rest = deposit(slice(0, h)), deposit(slice(h, n))
    # the sizes of a node's terms: |q| S for rho; a face's charge is at most |q| x the move in cells (< 0.1), the
    # ph current |q| x dph/dt (< 1), spread alike
    rho = deposit(slice(0, n), sign=False)[0].view(g.Nr + 1, g.ld)
    big = torch.nn.functional.max_pool2d(rho[None, None], 3, 1, 1)[0, 0].reshape(-1)
    dr, dth = float(g.rn[-1] - g.rn[-2]), float(g.tn[1] - g.tn[0])
    for k, scale in enumerate((1.0, 2 * dr / 1e-3, 2 * dth / 1e-3, 1.0)):
        err = (whole[k] - half[k] - rest[k]).abs()
        assert (err <= 2e4 * 2.0**-53 * scale * big).all(), (k, float((err / (scale * big + 1e-300)).max()))
