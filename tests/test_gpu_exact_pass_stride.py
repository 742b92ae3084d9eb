"""The mixed forms' exact pass over more tiles than its grid has CTAs (128 an
SM): deferred tiles (a phase beyond the head grid) at both ends of the grid's
stride, next to one another, one and many strides apart and in the ragged last
tile, against the float64 form on the same visibilities; the tiles between them
as well.

Tolerance: the mixed forms' bar, 1e-6 of the fluxes' sum.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu

dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")


@pytest.mark.parametrize("form", ["direct", "eq16", "eq17", "regrouped"])
def test_deferred_tiles_beyond_the_grid(form):
    ctas = 128 * torch.cuda.get_device_properties(0).multi_processor_count
    g = np.random.default_rng(7)
    l, m = g.uniform(-0.02, 0.02, (2, 3))
    f = np.array([1.0, 0.5, 0.25])
    n = 512 * ctas + 512 * 1000 + 77         # tiles of 512 visibilities at most
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    uvw = (torch.rand((n, 3), dtype=torch.float64, device="cuda", generator=gen) - 0.5) * 2e4
    far = [0, 3, 511, 512, 700, 512 * 7, 512 * ctas - 1, 512 * ctas, 512 * ctas + 700, 256 * ctas, 128 * ctas + 5,
           512 * (ctas + 900) + 3, n - 1]
    uvw[far] *= 500.0                        # millions of wavelengths: phases beyond 2^14 turns
    near = [min(max(k + d, 0), n - 1) for k in far for d in range(-300, 301, 20)]
    at = torch.tensor(sorted(set(near) | set(far) | set(range(11, n, 99991))), device="cuda")
    some = uvw[at].contiguous()
    if form == "direct":
        a = wt.dft_predict_vis(dev(l), dev(m), dev(f), uvw, mode=wt.WT_MIXED_FAST)[at]
        b = wt.dft_predict_vis(dev(l), dev(m), dev(f), some, mode=wt.WT_FP64)
    else:
        which = {"eq16": wt.WT_SUM_EQ16, "eq17": wt.WT_SUM_EQ17, "regrouped": wt.WT_SUM_EQ17_REGROUPED}[form]
        t = wt.wt_build_tree(dev(l), dev(m), dev(f), np.pi, np.pi / 4, 9)
        a = wt.wt_predict_vis(t, uvw, mode=wt.WT_MIXED_FAST, which=which)[at]
        b = wt.wt_predict_vis(t, some, mode=wt.WT_FP64, which=which)
    assert float((a - b).abs().max()) <= 1e-6 * f.sum()
