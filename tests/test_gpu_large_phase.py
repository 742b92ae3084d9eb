"""Float64 phases of 2^39 turns and more, up to where a float64 has no fraction
left: exact products (components at powers of two of l, whole u), so that the
phase is known to the last bit and the visibility is Eq. 12's plane wave at it.

Tolerance: 1e-12 of the flux; the sine and cosine are good to a few 2^-53.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_vis", [200, 40000])       # cut over its terms or not
@pytest.mark.parametrize("e", [20, 39, 40, 41, 42, 43, 47, 50, 53, 60])
def test_plane_wave_at_large_phases(e, n_vis):
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    g = np.random.default_rng(e)
    frac = g.integers(0, 32, n_vis) / 32.0            # in turns, dropped where t has no room for it
    t = g.choice([-1.0, 1.0], n_vis) * (2.0 ** e * g.integers(1, 2 ** 10, n_vis) / 2.0 ** 9 + frac)
    uvw = np.stack([t * 64.0, np.zeros(n_vis), np.zeros(n_vis)], axis=1)
    l, m, f = np.array([2.0 ** -6] * 300), np.zeros(300), np.ones(300)
    want = 300.0 * np.exp(2j * np.pi * np.remainder(t, 1.0))
    for sign in (1, -1):
        v = wt.dft_predict_vis(dev(l), dev(m), dev(f), dev(uvw), mode=wt.WT_FP64, sign=sign).cpu().numpy()
        assert np.max(np.abs(v - (want if sign > 0 else want.conj()))) <= 1e-12 * 300.0
