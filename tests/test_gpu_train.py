"""The fused training kernels against a plain torch restatement of the same
network: batches of one slice step, one chunk, several chunks and several
tiles per CTA."""
import pytest

from helpers import cuda_or_skip, fpic

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DIMS = (14, 128, 128, 128, 9)


def _bf(x):
    return x.to(torch.bfloat16).to(torch.float64)


def _reference(P, X, T, S, lw):
    """bf16 operands (weights, activations, dZ), exact sums."""
    W, b, o = [], [], 0
    for i, n in zip(DIMS[:-1], DIMS[1:]):
        W.append(_bf(P[o:o + n * i].view(n, i)))
        b.append(P[o + n * i:o + n * i + n].double())
        o += n * i + n
    H = [_bf(X[:, :14])]
    for k in range(3):
        H.append(_bf((H[-1] @ W[k].T + b[k]).clamp_min(0.0).float()))
    y = (H[3] @ W[3].T + b[3])
    d = 2.0 * lw * (y - T[:, :9].double())
    d[:, 6] = torch.sigmoid(y[:, 6]) - S.double()
    d = (d / X.shape[0]).float().double()
    out = []
    for k in (3, 2, 1, 0):
        out = [(_bf(d.float()).T @ H[k]).reshape(-1), d.sum(0)] + out
        if k:
            d = ((_bf(d.float()) @ W[k]) * (H[k] > 0)).float().double()
    return torch.cat(out)


@pytest.mark.parametrize("B", [256, 512, 2048, 8192, 65536])
def test_fused_gradient(B):
    """FP32 accumulation of exact bf16 products (relative 2^-24 sqrt(terms))
    and the odd activation or dZ whose bf16 rounding (2^-9) falls the other
    way, one in ~2^15 of a sum's terms: below 1e-3 of the gradient's norm."""
    cuda_or_skip()
    F = fpic()
    g = torch.Generator(device="cuda").manual_seed(B)
    rn = lambda *s: torch.randn(*s, generator=g, dtype=torch.float32, device="cuda")
    P = torch.cat([x for i, n in zip(DIMS[:-1], DIMS[1:]) for x in (rn(n * i) * (2.0 / i) ** 0.5, 0.1 * rn(n))])
    X = rn(B, 16)
    X[:, 14:] = 0.0
    T, S = rn(B, 16), (rn(B) > 0.5).float()
    lw = (1.0, 1.0, 0.5, 1.0, 2.0, 1.0, 0.0, 0.1, 0.3)
    net = F.MLP()
    net.set_params(P)
    _, got = net.grad(X, T, S, lw)
    assert net.status() == 0
    ref = _reference(P, X, T, S, torch.tensor(lw, dtype=torch.float64, device="cuda"))
    assert ((got.double() - ref).norm() / ref.norm()).item() <= 1e-3
    _, again = net.grad(X, T, S, lw)
    assert torch.equal(got, again)
