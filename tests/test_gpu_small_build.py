"""The one-CTA tree build (up to 1 024 components) at its edges, bit for bit
against the oracle's tree, and its records through the float64 Eq. 17 within
1e-10 of the oracle: component counts around warps and around the limit,
shallow and deep levels, repeated pixels, and the same components found through
a cross-reference table or imported as leaves.
"""
import numpy as np
import pytest

import oracle as O
import synth

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


@pytest.mark.parametrize("n", [1, 2, 31, 33, 700, 1023, 1024, 1025])
@pytest.mark.parametrize("J", [1, 2, 3, 9, 13, 30])
def test_tree_and_sum(n, J):
    g = np.random.default_rng(100 * n + J)
    l, m = g.uniform(-0.05, 0.05, (2, n))
    f = g.standard_normal(n)
    if n > 40:                                    # merged components, in input order
        at = g.integers(0, n // 3, n // 2)
        l[n - len(at):], m[n - len(at):] = l[at], m[at]
    t = wt.wt_build_tree(dev(l), dev(m), dev(f), synth.RA0, synth.DEC0, J)
    ot = O.Tree(l, m, f, synth.RA0, synth.DEC0, J)
    a, b = t.export(), ot.export()
    for k in ("key", "child_mask", "first_child", "lam", "gamma", "leaf_flux"):
        assert np.array_equal(a[k], b[k]), k
    uvw = g.uniform(-300, 300, (200, 3))
    v = wt.wt_predict_vis(t, dev(uvw)).cpu().numpy()
    assert np.max(np.abs(v - ot.vis_eq17(uvw))) <= 1e-10 * np.abs(f).sum()
    again = wt.wt_tree_import(a["key"][a["n_nodes"] - a["n_leaves"]:], a["leaf_flux"], synth.RA0, synth.DEC0, J)
    assert np.array_equal(wt.wt_predict_vis(again, dev(uvw)).cpu().numpy(), v)


@pytest.mark.parametrize("n", [5, 1024])
def test_through_the_table(n):
    g = np.random.default_rng(n)
    pix = g.integers(0, 256 * 256, n).astype(np.int32)
    f = g.standard_normal(n)
    table = wt.wt_xref_table(256, 1e-4, synth.RA0, synth.DEC0, 12)
    a = wt.wt_build_tree_xref(table, dev(pix), dev(f), synth.RA0, synth.DEC0, 12).export()
    l, m = (pix % 256 - 128) * 1e-4, (pix // 256 - 128) * 1e-4
    b = O.Tree(l, m, f, synth.RA0, synth.DEC0, 12).export()
    for k in ("key", "lam", "gamma", "leaf_flux"):
        assert np.array_equal(a[k], b[k]), k
