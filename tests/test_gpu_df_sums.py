"""The double-float direct sum's accumulation by itself: at baseline zero every
term is its flux, so that the sum's error against the exact total is that of the
additions alone.

Bar: the same sum with the double-float renormalised at every term (11 float32
operations each), emulated here step by step: blocks may not be worse, on the
average over many lists.
"""
import math

import numpy as np
import pytest

import oracle as O
import synth

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu


def _two_sum(a, b):
    s = a + b
    bp = s - a
    return s, (a - (s - bp)) + (b - bp)


def _renormalised_at_every_term(f):
    """[lists][terms] float64 -> [lists] float64."""
    h, l = np.zeros(len(f), np.float32), np.zeros(len(f), np.float32)
    for x in f.T:
        xh = x.astype(np.float32)
        xl = (x - xh.astype(np.float64)).astype(np.float32)
        s, e = _two_sum(h, xh)
        e = e + (l + xl)
        h = s + e
        l = e - (h - s)
    return h.astype(np.float64) + l.astype(np.float64)


@pytest.mark.parametrize("n", [20, 203, 1000])
def test_blocks_are_no_worse(n):
    g = np.random.default_rng(n)
    lists = 64
    f = 10.0 ** g.uniform(-3, 0, (lists, n))
    high = f.astype(np.float32).astype(np.float64)
    f = high + (f - high).astype(np.float32)              # exact as double-floats
    exact = np.array([math.fsum(x) for x in f])
    bar = _renormalised_at_every_term(f) - exact
    l, m = (torch.as_tensor(x, device="cuda") for x in g.uniform(-0.02, 0.02, (2, n)))
    uvw = torch.zeros((160000, 3), dtype=torch.float64, device="cuda")      # enough not to be cut over its terms
    got = np.empty(lists)
    for k in range(lists):
        v = wt.dft_predict_vis(l, m, torch.as_tensor(f[k], device="cuda"), uvw, mode=wt.WT_FP64_DF)
        assert float(v.imag.abs().max()) == 0.0 and bool((v == v[0]).all())
        got[k] = float(v[0].real)
    err = got - exact
    assert np.sqrt(np.mean((err / exact) ** 2)) <= np.sqrt(np.mean((bar / exact) ** 2))


@pytest.mark.parametrize("which", [wt.WT_SUM_EQ17_REGROUPED, wt.WT_SUM_EQ16])
@pytest.mark.parametrize("beyond", [-1, 0, 1, 70])
def test_shapes_without_tuning(which, beyond, monkeypatch):
    """At the line where the default turns to pairs of visibilities; the form's
    bar, 1e-10 of the fluxes' sum, against the oracle's sums."""
    monkeypatch.setenv("WT_AUTOTUNE", "0")
    n = 2 * 128 * torch.cuda.get_device_properties(0).multi_processor_count + beyond
    g = np.random.default_rng(3)
    l, m = g.uniform(-0.01, 0.01, (2, 40))
    f = g.uniform(0.5, 1.5, 40)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    t = wt.wt_build_tree(dev(l), dev(m), dev(f), synth.RA0, synth.DEC0, 9)
    uvw = g.uniform(-1000, 1000, (n, 3))
    v = wt.wt_predict_vis(t, dev(uvw), mode=wt.WT_FP64_DF, which=which).cpu().numpy()
    at = np.r_[0:300, n - 300:n]
    ref = O.Tree(l, m, f, synth.RA0, synth.DEC0, 9).vis_eq17(uvw[at], 1)
    assert np.max(np.abs(v[at] - ref)) <= 1e-10 * f.sum()
