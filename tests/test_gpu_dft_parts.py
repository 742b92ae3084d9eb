"""The direct sum cut over its terms (few visibilities, many components),
against the same sum with every visibility repeated until the tiles alone fill
the chip, which is not cut: the same terms in another order of addition.

Tolerance: float64 sums of n terms of |C| <= 1 differ by at most 2 n 2^-53
Sigma|C|, double-float ones (2^-47 per addition) likewise; the mixed forms add
blocks of 8 in float32 and compensate between them, 8 2^-24 of a block's
magnitude each way, so 2^-20 Sigma|C| covers both sides.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu

MODES = {"fp64": wt.WT_FP64, "df": wt.WT_FP64_DF, "mixed": wt.WT_MIXED, "fast": wt.WT_MIXED_FAST,
         "tc": wt.WT_MIXED_TC}


@pytest.mark.parametrize("mode", sorted(MODES))
@pytest.mark.parametrize("n_vis,n_comp", [(1, 1000), (127, 129), (129, 4096), (513, 20000), (8128, 5000),
                                          (20011, 641)])
def test_cut_sum_equals_the_whole(mode, n_vis, n_comp):
    g = np.random.default_rng(n_vis + n_comp)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    l, m = g.uniform(-0.02, 0.02, (2, n_comp))
    f = 10.0 ** g.uniform(-3, 0, n_comp)
    uvw = g.uniform(-2e4, 2e4, (n_vis, 3))
    if mode in ("mixed", "fast", "tc"):
        uvw[n_vis // 2] *= 100        # beyond the head grid: its tile takes the exact pass
    a = wt.dft_predict_vis(dev(l), dev(m), dev(f), dev(uvw), mode=MODES[mode], sign=-1)
    reps = 1 + 700 * 512 // n_vis
    b = wt.dft_predict_vis(dev(l), dev(m), dev(f), dev(uvw).repeat(reps, 1), mode=MODES[mode], sign=-1)[:n_vis]
    tol = {"fp64": 2.0 ** -52 * n_comp, "df": 2.0 ** -46 * n_comp}.get(mode, 2.0 ** -20)
    assert float((a - b).abs().max()) <= tol * f.sum()


@pytest.mark.parametrize("n_vis", [1, 300, 8128])
def test_cut_leaf_sum_on_the_tensor_cores(n_vis):
    g = np.random.default_rng(n_vis)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    l, m = g.uniform(-0.02, 0.02, (2, 3000))
    f = 10.0 ** g.uniform(-3, 0, 3000)
    uvw = dev(g.uniform(-2e4, 2e4, (n_vis, 3)))
    t = wt.wt_build_tree(dev(l), dev(m), dev(f), np.pi, np.pi / 4, 12)
    a = wt.wt_predict_vis(t, uvw, mode=wt.WT_MIXED_TC, which=wt.WT_SUM_EQ16)
    b = wt.wt_predict_vis(t, uvw.repeat(1 + 700 * 128 // n_vis, 1), mode=wt.WT_MIXED_TC, which=wt.WT_SUM_EQ16)[:n_vis]
    assert float((a - b).abs().max()) <= 2.0 ** -20 * f.sum()
