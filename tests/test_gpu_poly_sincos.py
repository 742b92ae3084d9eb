"""The polynomial form's sine and cosine: the error of single plane waves of unit
flux against float64, over millions of phases spread evenly over the turn.

Bar: the error of Taylor series to x^9 and x^10 in the same float32 steps, by an
emulation of them over 4e7 phases: 2.034e-8 RMS, 9.97e-8 at most. A polynomial
form of fewer terms has to be as good. (The phase itself, in double-float, is
good to 1e-13 of a turn here, and one term's sum adds no rounding.)
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sign", [1, -1])
def test_error_of_unit_waves(sign):
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    n = 1 << 22
    uvw = (torch.rand((n, 3), dtype=torch.float64, device="cuda", generator=g) - 0.5) * 1e4
    l, m = 0.0123456789, -0.0087654321
    nm1 = -(l * l + m * m) / (1.0 + np.sqrt(1.0 - (l * l + m * m)))
    t = uvw[:, 0] * l + uvw[:, 1] * m + uvw[:, 2] * nm1
    t = (t - torch.round(t)) * (2.0 * np.pi * sign)
    one = lambda x: torch.tensor([x], dtype=torch.float64, device="cuda")
    v = wt.dft_predict_vis(one(l), one(m), one(1.0), uvw, mode=wt.WT_MIXED, sign=sign)
    e = torch.view_as_real(v).double() - torch.stack([torch.cos(t), torch.sin(t)], dim=1)
    assert float(e.abs().max()) <= 1.0e-7
    assert float((e * e).mean().sqrt()) <= 2.034e-8
