"""The batched persistent clean against the one-launch-per-component schedule on
images with pixels of plus infinity, bit for bit (fluxes of infinity, the NaN
that infinity less infinity leaves, the infinities that its beam spreads).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("low", [0.0, 0.05])          # a beam with zeros, or with sidelobes of both signs
@pytest.mark.parametrize("n", [4, 62, 128, 150, 258])
def test_infinite_pixels(n, low, monkeypatch):
    g = np.random.default_rng(n)
    img = g.standard_normal((n, n)).astype(np.float32)
    img[g.integers(0, n, 3), g.integers(0, n, 3)] = np.inf
    img[0, n - 1] = -np.inf
    psf = (low * g.uniform(-1, 1, (n, n))).astype(np.float32)
    psf[n // 2, n // 2] = 1.0
    out = []
    for launches in (False, True):
        if launches:
            monkeypatch.setenv("WT_HOGBOM", "launches")
        else:
            monkeypatch.delenv("WT_HOGBOM", raising=False)
        w = torch.as_tensor(img, device="cuda").clone()
        pix, flux = wt.wt_hogbom(w, torch.as_tensor(psf, device="cuda"), 0.2, 100, -10.0)
        out.append([x.cpu().numpy().view(np.uint32) for x in (w, pix, flux)])
    assert len(out[0][1]) >= 1
    for a, b in zip(*out):
        assert np.array_equal(a, b)
