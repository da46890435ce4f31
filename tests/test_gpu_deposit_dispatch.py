"""Which form the deposit takes: per-cell polynomials on fine grids, built by the
first deposit on a grid; lattices on coarse ones and in a first deposit that is
being captured; and the tables of the grid a context has now."""
import numpy as np
import pytest

from paper_2602_07452_gb300 import inputs as I
from helpers import cuda_or_skip, fpic, make_particles

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
A = 0.9


def _grid(side):
    return I.log_grid(side, side, 0.9 * I.horizon(1.0, A), 50.0)


def _particles(g, n=20000, seed=1):
    rng = np.random.default_rng(seed)
    z = np.zeros((n, 6))
    z[:, 0] = np.exp(rng.uniform(np.log(1.6), np.log(45.0), n))
    z[:, 1] = rng.uniform(0.02, np.pi - 0.02, n)
    z[:, 3:] = rng.normal(size=(n, 3))
    return z, rng.choice([-1.0, 1.0], n), rng.uniform(0.5, 2.0, n)


def _deposit(F, ctx, g):
    z, q, w = _particles(g)
    return torch.stack(F.fpic_deposit(ctx, make_particles(z, q, w=w), g.size))


def _fresh(F, g):
    ctx = F.fpic_init_metric(1.0, A)
    F.fpic_set_grid(ctx, g)
    return _deposit(F, ctx, g)


@pytest.mark.parametrize("side,poly", [(300, True), (100, False)])
def test_first_deposit_under_capture_takes_the_lattices(side, poly):
    """Scratch in place from a larger grid; the first deposit on this one captured
    and replayed, then one outside: other bits where the polynomials serve (to the
    pairs' accuracy, 1e-12 of the largest source), the same where they do not; and
    the graph replays to its own bits afterwards."""
    cuda_or_skip()
    F = fpic()
    ctx = F.fpic_init_metric(1.0, A)
    big, g = _grid(320), _grid(side)
    F.fpic_set_grid(ctx, big)
    _deposit(F, ctx, big)
    F.fpic_set_grid(ctx, g)
    z, q, w = _particles(g)
    p = make_particles(z, q, w=w)
    out = tuple(torch.zeros(g.size, dtype=torch.float64, device="cuda") for _ in range(4))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        F.fpic_deposit(ctx, p, g.size, out=out)
    graph.replay()
    torch.cuda.synchronize()
    captured = torch.stack(out).clone()
    later = _deposit(F, ctx, g)
    assert torch.equal(captured, later) != poly
    assert ((captured - later).abs().amax(1) <= 1e-12 * later.abs().amax(1)).all()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(torch.stack(out), captured)


def test_tables_follow_the_grid():
    """One context moved between fine and coarse grids: the bits of a fresh one."""
    cuda_or_skip()
    F = fpic()
    ctx = F.fpic_init_metric(1.0, A)
    for side in (256, 90, 320, 256):
        g = _grid(side)
        F.fpic_set_grid(ctx, g)
        assert torch.equal(_deposit(F, ctx, g), _fresh(F, g)), side
