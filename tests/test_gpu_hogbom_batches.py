"""The batched persistent clean against the one-launch-per-component schedule,
bit for bit: image, components and fluxes. Images where many pixels compete
(noise, ties, constants), beams whose sidelobes raise other pixels, high and
low gains, a threshold that stops the clean inside a batch, sizes around the
128-pixel segments and the SM count, NaN and infinite pixels.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu


def _both(img, psf, gain, iters, threshold, monkeypatch):
    out = []
    for launches in (False, True):
        if launches:
            monkeypatch.setenv("WT_HOGBOM", "launches")
        else:
            monkeypatch.delenv("WT_HOGBOM", raising=False)
        w = torch.as_tensor(img, device="cuda").clone()
        pix, flux = wt.wt_hogbom(w, torch.as_tensor(psf, device="cuda"), gain, iters, threshold)
        out.append((w.cpu().numpy(), pix.cpu().numpy(), flux.cpu().numpy()))
    return out


def _beam(n, g, low):
    y, x = np.mgrid[0:n, 0:n] - n // 2
    r2 = (x * x + y * y).astype(np.float64)
    b = np.exp(-r2 / 3.0) + low * g.uniform(-1, 1, (n, n))
    b[n // 2, n // 2] = 1.0
    return b.astype(np.float32)


@pytest.mark.parametrize("n", [2, 4, 62, 126, 128, 130, 150, 154, 258, 642])
@pytest.mark.parametrize("kind", ["sources", "noise", "ties", "odd"])
def test_batches_equal_single_components(n, kind, monkeypatch):
    g = np.random.default_rng(n)
    low, gain, iters, thr = 0.02, 0.1, 300, 0.0
    if kind == "sources":
        img = np.zeros((n, n))
        img[g.integers(0, n, 40), g.integers(0, n, 40)] += 10.0 ** g.uniform(-1, 0.5, 40)
        img += 0.01 * g.standard_normal((n, n))
        thr = 0.05
    elif kind == "noise":
        img, low, gain = g.standard_normal((n, n)), 0.3, 1.0
    elif kind == "ties":
        img, low, thr = g.integers(-3, 4, (n, n)) / 4.0, 0.0, -10.0
    else:
        img, thr = -np.abs(g.standard_normal((n, n))), -5.0
        img[n // 2, n // 2] = np.nan
        if n > 4:
            img[1, 2] = -np.inf
    a, b = _both(img.astype(np.float32), _beam(n, g, low), gain, iters, thr, monkeypatch)
    for x, y in zip(a, b):
        assert x.shape == y.shape and np.array_equal(x.view(np.uint32), y.view(np.uint32))
