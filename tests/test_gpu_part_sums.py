"""The direct sum cut over its terms, mixed forms: the parts' sums are added with
nothing rounded off them, and the whole is within the forms' bars of the oracle's
Eq. 12.

At baseline zero every term is its flux. With whole fluxes below 2^20 a block of
eight is exact in float32 and so is the compensated sum of the blocks, so the
visibility is the exact total, rounded to float32 once: equality. (A part's sum,
of the order of 2^27, is no float32 by itself: rounded, one total in ten or so
comes out elsewhere.)
"""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu

MODES = {"mixed": wt.WT_MIXED, "fast": wt.WT_MIXED_FAST, "tc": wt.WT_MIXED_TC}
dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")


@pytest.mark.parametrize("n_comp", [300, 512])
@pytest.mark.parametrize("mode", sorted(MODES))
def test_parts_are_not_rounded(mode, n_comp):
    uvw = dev(np.zeros((130, 3)))
    for seed in range(64):
        g = np.random.default_rng(seed)
        l, m = g.uniform(-0.02, 0.02, (2, n_comp))
        f = g.integers(2 ** 19, 2 ** 20, n_comp).astype(np.float64)
        v = wt.dft_predict_vis(dev(l), dev(m), dev(f), uvw, mode=MODES[mode]).cpu().numpy()
        assert np.array_equal(v, np.full(130, np.float32(f.sum()), dtype=np.complex64)), seed


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("n_vis,n_comp", [(1, 300), (129, 1000), (780, 3760)])
@pytest.mark.parametrize("mode", ["fp64", "df"] + sorted(MODES))
def test_cut_sum_against_the_oracle(mode, n_vis, n_comp, sign):
    g = np.random.default_rng(n_vis)
    l, m = g.uniform(-0.02, 0.02, (2, n_comp))
    f = 10.0 ** g.uniform(-3, 0, n_comp)
    uvw = g.uniform(-2e4, 2e4, (n_vis, 3))
    if mode in MODES:
        uvw[n_vis // 2] *= 100           # beyond the head grid: its tile takes the exact pass
    which = {"fp64": wt.WT_FP64, "df": wt.WT_FP64_DF, **MODES}[mode]
    v = wt.dft_predict_vis(dev(l), dev(m), dev(f), dev(uvw), mode=which, sign=sign).cpu().numpy()
    tol = 1e-10 if mode in ("fp64", "df") else 1e-6
    assert np.max(np.abs(v - O.dft(l, m, f, uvw, sign))) <= tol * f.sum()
