"""Every sample of a training batch counts once, those at the edges of the
64-sample tiles, of the grid and of a minibatch that wraps around above all.

The targets are the network's own outputs (float64, with the two documented
bfloat16 roundings) but for one sample, whose residual is (1, -1/2): it carries
the loss and the gradient, so that losing it, or taking it twice, is an error of
the order of one.

Tolerance: 0.05. The other samples' residuals are the float32 forward pass's
errors, 1e-6, and those of hidden units that round to the other bfloat16, 1e-4 on
some tens of samples: together below 1e-2 of the one sample's share.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu

LEVEL = 11
SCALE = float(np.float32(np.sqrt(np.pi / 3) * 2.0 ** (1 - LEVEL)))


def _unpack(p):
    out, at = [], 0
    for shape in ((64, 3), (64,), (64, 64), (64,), (2, 64), (2,)):
        n = int(np.prod(shape))
        out.append(p[at:at + n].reshape(shape))
        at += n
    return out


def _outputs(p, x):
    w1, b1, w2, b2, w3, b3 = _unpack(p)
    rnd = lambda z: z + (z.detach().to(torch.bfloat16).to(torch.float64) - z.detach())
    silu = torch.nn.functional.silu
    return silu(rnd(silu(x @ w1.T + b1)) @ rnd(w2).T + b2) @ w3.T + b3


def _network(n):
    m = wt.Mlp(LEVEL, np.pi, np.pi / 4, depth=2, x_max=1e30, seed=n)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    x = torch.rand((n, 3), dtype=torch.float64, device="cuda", generator=g) * 8 - 4
    p = torch.as_tensor(m.get_params(), dtype=torch.float64, device="cuda")
    return m, x, _outputs(p, x).to(torch.float32), p


@pytest.mark.parametrize("n", [1, 63, 64, 65, 130, 304 * 64, 304 * 64 + 1, 20011, 2 * 304 * 64 + 65])
def test_every_edge_sample_counts_once(n):
    m, x, y, p = _network(n)
    grid = 64 * 2 * torch.cuda.get_device_properties(0).multi_processor_count
    edges = {0, 63, 64, 65, grid - 1, grid, grid + 63, grid + 64, 2 * grid - 1, 2 * grid, 2 * grid + 64, n - 1}
    for k in sorted(e for e in edges if 0 <= e < n):
        t = y.clone()
        t[k] += torch.tensor([1.0, -0.5], device="cuda")
        loss, grad = m.loss_grad(x / SCALE, t)
        assert abs(loss * n / 1.25 - 1.0) <= 0.05, k
        q = p.clone().requires_grad_(True)
        e = ((_outputs(q, x[k:k + 1]) - t[k].to(torch.float64)) ** 2).sum() / n
        want = torch.autograd.grad(e, q)[0].cpu().numpy()
        at = 0
        for size in (192, 64, 4096, 64, 128, 2):
            a, b = grad[at:at + size], want[at:at + size]
            assert np.linalg.norm(a - b) <= 0.05 * np.linalg.norm(b), (k, at)
            at += size


@pytest.mark.parametrize("n,batch,step", [(1000, 300, 3), (1000, 300, 0), (700, 700, 2), (500, 129, 11)])
def test_a_minibatch_that_wraps_around(n, batch, step):
    m, x, y, _ = _network(n)
    state = m.get_state()
    first = step * batch % n
    inside = {(first + i) % n for i in range(batch)}
    for k in {first, (first + batch - 1) % n, 0, n - 1, (first + batch) % n, (first - 1) % n}:
        t = y.clone()
        t[k] += torch.tensor([1.0, -0.5], device="cuda")
        m.set_state(*state)
        loss = m.train_range(x / SCALE, t, step, 1, 100, batch=batch)
        want = 1.25 if k in inside else 0.0
        assert abs(loss * batch - want) <= 0.05, k
