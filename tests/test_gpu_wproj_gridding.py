"""The w-projection gridding itself, against its definition in float64.

wt_dirty_image_w approximates the w-corrected image (test_gpu_wproj.py holds
it to the direct sum); here the approximation is taken as given -- the tabulated
kernel at 8 points per cell, the nearest table point found in single precision
for each tap of each of a visibility's two entries, linear interpolation
between planes, each entry's own support -- and evaluated in float64, so that
what is left is rounding. Offsets at and around the ties between two table
points, supports that touch the grid's border and both signs of w are among
the visibilities.

Tolerance: image times grid correction, a sum over all taps of |V| |K| / W
terms. A tap carries the float32 table (2^-24 and its two sums of 64, 2^-21
together), interpolation, product and accumulation over at most 80 entries
(some 2^-22), and the transform log2(n^2) = 14 roundings: 2^-19 of the sum of
the terms' magnitudes covers them.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
wt = pytest.importorskip("paper_1909_03956_gb300")

pytestmark = pytest.mark.gpu

WIDTH, BETA, OVER, M = 7, 16.25, 8, 128


def _kb(t):
    a = BETA ** 2 - (np.pi * WIDTH * t) ** 2
    r = np.sqrt(np.abs(a))
    return np.where(a > 0, np.sinh(r), np.sin(r)) / r / (np.sinh(BETA) / BETA)


def _reference(uvw, vis, n, dl, planes):
    """Image times grid correction, and the bound on its terms' sum."""
    ndl = n * dl
    per_w = ndl * ndl / (2 * np.sqrt(1 - 0.5 * ndl * ndl))
    w_max = np.abs(uvw[:, 2]).max()
    h = int(np.ceil(0.5 * WIDTH + w_max * per_w)) + 1
    dw = w_max / (planes - 1)
    t = (np.arange(M) + 0.5) / M - 0.5
    r2 = (t * ndl)[:, None] ** 2 + (t * ndl)[None, :] ** 2
    nm1 = -r2 / (1 + np.sqrt(1 - r2))
    T = (2 * h + 1) * OVER + 1
    tw = np.exp(2j * np.pi * (np.arange(T) / OVER - (h + 0.5))[:, None] * t[None, :])
    K = [tw @ (np.outer(_kb(t), _kb(t)) * np.exp(-2j * np.pi * p * dw * nm1)) @ tw.T / M ** 2 for p in range(planes)]
    grid = np.zeros((n, n), dtype=complex)
    mass, entries = 0.0, 0
    half = n // 2

    def index(d, f):       # single precision, as documented
        x = (np.float32(d) - np.float32(f)) + np.float32(h) + np.float32(0.5)
        return int(np.rint(np.float32(x * np.float32(OVER))))

    for (u, v, w), V in zip(uvw, vis):
        if abs(np.rint(u * ndl)) > half - h - 1 or abs(np.rint(v * ndl)) > half - h - 1:
            continue
        entries += 2
        for s in (1, -1):
            x, y, ww, Z = s * u * ndl, s * v * ndl, s * w, V if s == 1 else np.conj(V)
            ic, jc = int(np.rint(x)), int(np.rint(y))
            he = min(h, int(np.ceil(0.5 * WIDTH + per_w * abs(ww))) + 1)
            p = min(int(abs(ww) / dw), planes - 2)
            a = min(max(abs(ww) / dw - p, 0.0), 1.0)
            for dx in range(-he, he + 1):
                ix = index(dx, x - ic)
                for dy in range(-he, he + 1):
                    jx, jy = ix, index(dy, y - jc)
                    if ww < 0:
                        jx, jy = T - 1 - jx, T - 1 - jy
                    k = K[p][jx, jy] + a * (K[p + 1][jx, jy] - K[p][jx, jy])
                    k = np.conj(k) if ww < 0 else k
                    grid[(jc + dy) % n, (ic + dx) % n] += Z * k
                    mass += abs(Z) * abs(k)
    return np.fft.fftshift(np.fft.fft2(grid)).real / entries, mass / entries


@pytest.mark.parametrize("n,planes,w_scale", [(128, 2, 3000.0), (128, 16, 30000.0), (130, 9, 30000.0), (96, 5, 10.0)])
def test_gridding_equals_its_definition(n, planes, w_scale):
    rng = np.random.default_rng(n + planes)
    dl = 2.0 ** -13
    lim = n // 2 - 10
    x = rng.uniform(-lim, lim, (80, 2))
    x[:30] = np.rint(x[:30]) + (2 * rng.integers(-4, 4, (30, 2)) + 1) / 16      # between two table points
    x[10:20] += rng.choice([-1e-7, 1e-7, -1e-6, 1e-6], (10, 2))
    x[30:34] = [[lim + 9.4, 0], [0, -lim - 9.4], [-lim, lim], [lim + 0.49, -lim - 0.49]]   # border, off the grid
    uvw = np.column_stack([x / (n * dl), rng.uniform(-w_scale, w_scale, 80)])
    vis = (rng.standard_normal(80) + 1j * rng.standard_normal(80)).astype(np.complex64)
    img = wt.wt_dirty_image_w(torch.as_tensor(uvw, device="cuda"), torch.as_tensor(vis, device="cuda"), n, dl,
                              w_planes=planes).cpu().numpy().astype(np.float64)
    ref, mass = _reference(uvw, vis.astype(complex), n, dl, planes)
    c = _kb((np.arange(n) - n // 2) / n)
    err = np.abs(img * np.outer(c, c) - ref).max()
    assert err <= 2.0 ** -19 * mass, (err, mass)
