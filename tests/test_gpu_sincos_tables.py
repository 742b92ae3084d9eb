"""The table sines and cosines of the float64 and double-float forms: one
component of unit flux, so that each visibility is exp(i 2 pi t) itself, at
phases on, beside and between the 1 024 table points, on both sides of a turn
and far from it.

The component sits at l = 2^-4, m = 0, w = 0, so t = u / 16 exactly. Float64:
the reduction is exact; table entry, two inner roundings and the result's err
by at most 2^-53 each, twice over for the products: 4 2^-53. Double-float: the
phase carries 48 bits of |t| (2^-46 |t| turns, 2 pi as an angle) and the
rotation some 8 roundings of 2^-48.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu


def _phases():
    k = np.arange(-1024, 1025)
    t = np.concatenate([k / 1024, (k + 0.5) / 1024, np.nextafter((k + 0.5) / 1024, 9), (k + 0.4999) / 1024,
                        k / 1024 + 2.0 ** -40, k + 0.125, 517.3 * k / 1024, k * 31.999 / 2, [0.0, -0.0, 0.25, 0.5]])
    return t


@pytest.mark.parametrize("mode", ["fp64", "df"])
@pytest.mark.parametrize("sign", [1, -1])
def test_single_component_phases(mode, sign):
    t = _phases()
    uvw = np.zeros((len(t), 3))
    uvw[:, 0] = 16.0 * t
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    v = wt.dft_predict_vis(dev(np.array([0.0625])), dev(np.array([0.0])), dev(np.array([1.0])), dev(uvw),
                           mode=wt.WT_FP64 if mode == "fp64" else wt.WT_FP64_DF, sign=sign).cpu().numpy()
    f = t - np.rint(t)
    ref = np.cos(2 * np.pi * f.astype(np.longdouble)) + 1j * sign * np.sin(2 * np.pi * f.astype(np.longdouble))
    tol = 4 * 2.0 ** -53 if mode == "fp64" else 2 * np.pi * 2.0 ** -46 * np.abs(t) + 8 * 2.0 ** -48
    tol = tol + 2 * np.pi * np.abs(f) * 2.0 ** -53 * (np.finfo(np.longdouble).eps > 2.0 ** -60)   # the reference's own
    assert np.all(np.abs(v - ref.astype(complex)) <= tol + 2.0 ** -53)
