"""The float64 Eq. 17 takes a run of sibling leaves and their parent as one step
where they lie in one staging chunk (64 records), two leaves at a time
elsewhere: trees whose runs (one to four leaves, every set of child slots) fall
at every place against the chunks' edges, against the oracle's Eq. 17.

Tolerance: the float64 form's bar, 1e-10 of the fluxes' sum. A leaf in another
slot or left out changes the sum by its own share, 1e-3 at least.
"""
import numpy as np
import pytest

import oracle as O
import synth

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_vis", [63, 130])
@pytest.mark.parametrize("n", [3, 40, 97, 150, 151, 152, 153, 154, 155, 156, 157, 400])
def test_runs_of_siblings_at_chunk_edges(n, n_vis):
    g = np.random.default_rng(n)
    # level-9 pixels are 4e-3 rad wide: a field of a few dozen to a few hundred
    # of them, filled in part, has runs of every length
    half = 2e-3 * np.sqrt(2.0 * n)
    l, m = g.uniform(-half, half, (2, n))
    f = g.uniform(0.5, 1.5, n)
    J = 9
    ot = O.Tree(l, m, f, synth.RA0, synth.DEC0, J)
    runs = {bin(int(x)).count("1") for x in ot.export()["child_mask"]}
    assert n < 97 or runs >= {0, 1, 2, 3, 4}
    t = wt.wt_build_tree(*(torch.as_tensor(a, device="cuda") for a in (l, m, f)), synth.RA0, synth.DEC0, J)
    uvw = g.uniform(-300, 300, (n_vis, 3))
    for sign in (1, -1):
        v = wt.wt_predict_vis(t, torch.as_tensor(uvw, device="cuda"), mode=wt.WT_FP64, sign=sign,
                              which=wt.WT_SUM_EQ17).cpu().numpy()
        assert np.max(np.abs(v - ot.vis_eq17(uvw, sign))) <= 1e-10 * f.sum()
