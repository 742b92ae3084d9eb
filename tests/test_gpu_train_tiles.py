"""Loss and gradient of the response network at the edges of the training
kernel's 64-sample tiles and of its grid, against float64 with the two
documented bfloat16 roundings (W2 and the first hidden layer).

Tolerance. The kernel's float32 sums err by 1e-6 at most; what dominates is a
hidden unit whose float32 value rounds to the other bfloat16: a share of about
2^-12 of the units (float32 errors of a few 2^-24 against a spacing of 2^-9),
each changing its products by 2^-8, so 2^-8 2^-6 = 6e-5 of a sum over many
samples; four times that, or one such unit of a row (2^-8 / sqrt(64)) twice
over for a single tile. A sample lost or taken twice among n shows as about
n^-1/2, 7e-3 at the largest n here.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu


def _reference(params, x, t):
    p = torch.as_tensor(params, dtype=torch.float64, device="cuda").requires_grad_(True)
    cut, at = [], 0
    for shape in ((64, 3), (64,), (64, 64), (64,), (2, 64), (2,)):
        n = int(np.prod(shape))
        cut.append(p[at:at + n].reshape(shape))
        at += n
    w1, b1, w2, b2, w3, b3 = cut
    rnd = lambda z: z + (z.detach().to(torch.bfloat16).to(torch.float64) - z.detach())
    silu = torch.nn.functional.silu
    y = silu(rnd(silu(x @ w1.T + b1)) @ rnd(w2).T + b2) @ w3.T + b3
    loss = ((y - t) ** 2).sum() / x.shape[0]
    return float(loss), torch.autograd.grad(loss, p)[0].cpu().numpy()


@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 8192, 304 * 32, 304 * 32 + 1, 304 * 64 + 1, 20011])
def test_loss_and_gradient_at_tile_edges(n):
    level = 11
    m = wt.Mlp(level, np.pi, np.pi / 4, depth=2, x_max=1e30, seed=n)
    scale = float(np.float32(np.sqrt(np.pi / 3) * 2.0 ** (1 - level)))
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    x = torch.rand((n, 3), dtype=torch.float64, device="cuda", generator=g) * 8 - 4
    t = torch.rand((n, 2), dtype=torch.float32, device="cuda", generator=g)
    loss, grad = m.loss_grad(x / scale, t)
    l0, g0 = _reference(m.get_params(), x, t.to(torch.float64))
    tol = 1e-3 if n <= 64 else 2.5e-4
    assert abs(loss - l0) <= tol * l0
    at = 0
    for size in (192, 64, 4096, 64, 128, 2):
        a, b = grad[at:at + size], g0[at:at + size]
        assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b), at
        at += size
