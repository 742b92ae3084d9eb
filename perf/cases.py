"""The work a user of this framework has it do, as cases that can be timed and compared.

Kinds of case, each through the entry points a program calls:

    cycle      one major cycle's model side: build the tree from the component list, predict, subtract
    predict    visibilities from a tree in hand (wt_predict_vis)
    direct     the direct sum over the components (dft_predict_vis)
    batched    many channels with trees of their own in one call (wt_predict_vis_batched)
    image      the dirty image of a set of visibilities, with w-projection or nearest-cell
    clean      Hogbom minor cycles on a dirty image (wt_hogbom)
    train      a stage of a response network's training (Mlp.train from given parameters)
    truncated  the tree cut at a level, its pixels' responses from a network (wt_predict_vis_truncated)

The arrays, skies and sizes are those of the repository's synthetic workloads (antennas uniform in a disc, components
uniform or in Gaussian blobs, log-uniform fluxes) and of its benchmark; the draws spread over the ranges between them.
"""
import math

import numpy as np
import torch

import paper_1909_03956_gb300 as wt

C_LIGHT = 299792458.0
LAT = math.radians(34.0784)
RA0, DEC0 = math.pi, math.radians(45.0)
FREQ = 1.4e9
MODES = {"fp64": wt.WT_FP64, "df": wt.WT_FP64_DF, "mixed": wt.WT_MIXED, "fast": wt.WT_MIXED_FAST, "tc": wt.WT_MIXED_TC}
SUMS = {"eq17": wt.WT_SUM_EQ17, "regrouped": wt.WT_SUM_EQ17_REGROUPED, "eq16": wt.WT_SUM_EQ16}


def listed():
    return [
        # The smallest major cycle: a 32-antenna array, ten thousand visibilities, a hundred components, in the default
        # mode and sum (float64, Eq. 17). Launches and the tree build weigh most.
        dict(name="cycle_small", kind="cycle", n_ant=32, diameter=2000.0, n_times=20, drop=0, n_comp=100, blobs=0,
             field=1.0, J=8, mode="fp64", sum="eq17", sign=1),
        # The benchmark's step: 16 M visibilities, 50 000 clustered components, the form the README recommends.
        dict(name="cycle_large", kind="cycle", n_ant=256, diameter=10000.0, n_times=490, drop=0, n_comp=50000,
             blobs=20, field=2.0, J=12, mode="fast", sum="regrouped", sign=1),
        # wt_predict_vis with its defaults on an hour of a 64-antenna array, a ragged count left by flagging.
        dict(name="predict_defaults", kind="predict", n_ant=64, diameter=5000.0, n_times=100, drop=37, n_comp=5000,
             blobs=20, field=2.0, J=12, mode="fp64", sum="eq17", sign=1),
        # The mixed-precision configuration, one channel, the default sum, the conjugate convention.
        dict(name="predict_mixed", kind="predict", n_ant=128, diameter=10000.0, n_times=250, drop=0, n_comp=20000,
             blobs=20, field=2.0, J=12, mode="mixed", sum="eq17", sign=-1),
        # Float64-class accuracy on the float32 pipe: the medium array.
        dict(name="predict_df", kind="predict", n_ant=64, diameter=5000.0, n_times=500, drop=0, n_comp=5000, blobs=20,
             field=2.0, J=12, mode="df", sum="regrouped", sign=1),
        # One integration of a 128-antenna array against a whole component list in the default mode: what calibration
        # asks for time step by time step.
        dict(name="direct_snapshot", kind="direct", n_ant=128, diameter=10000.0, n_times=1, drop=0, n_comp=5000,
             blobs=20, field=2.0, mode="fp64", sign=1),
        # The direct sum of the medium array, phases on the tensor cores.
        dict(name="direct_tc", kind="direct", n_ant=64, diameter=5000.0, n_times=500, drop=0, n_comp=5000, blobs=20,
             field=2.0, mode="tc", sign=1),
        # A quarter of the 64-channel workload: uneven trees, J = 10 .. 13, one call.
        dict(name="batched", kind="batched", n_ant=128, diameter=10000.0, n_times=62, drop=0, n_ch=16, n_comp=20000,
             blobs=20, field=2.0, J_lo=10, J_hi=13, mode="fast", sign=1),
        # The wide-field dirty image of a major cycle: the medium array at 2048 x 2048, 64 w-planes.
        dict(name="image_w", kind="image", n_ant=64, diameter=5000.0, n_times=500, drop=0, n=2048, dl=2.1e-5,
             planes=64),
        # The minor cycles of one major cycle: a thousand components off a 2048 x 2048 image.
        dict(name="clean", kind="clean", n=2048, iters=1000, gain=0.1, sources=300),
        # A stage of a response network's training, the benchmark's batch and rate.
        dict(name="train", kind="train", samples=500000, batch=8192, steps=24, lr=3e-3, x_span=46.0),
        # The learned form on the large workload: the tree cut at level 11.
        dict(name="truncated_learned", kind="truncated", n_ant=256, diameter=10000.0, n_times=490, drop=0,
             n_comp=50000, blobs=20, field=2.0, J=12, level=11, sign=1),
    ]


# Term rates (per second) that bound a drawn case's cost by the largest listed one's.
RATES = {"fp64": 1.2e10, "df": 1.0e11, "mixed": 2.0e11, "fast": 6.0e11, "tc": 1.5e12}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _array(rng, n_vis_hi, n_vis_lo=1000):
    """Antennas, extent and times of an array with between n_vis_lo and n_vis_hi visibilities, an odd few dropped."""
    want = _log(rng, n_vis_lo, max(n_vis_lo + 1, n_vis_hi))
    n_ant = rng.randint(20, 256)
    while n_ant * (n_ant - 1) // 2 > want and n_ant > 20:
        n_ant = max(20, int(n_ant * 0.8))
    per = n_ant * (n_ant - 1) // 2
    return dict(n_ant=n_ant, diameter=float(rng.choice([2000, 3400, 5000, 10000])), n_times=max(1, want // per),
                drop=rng.choice([0, 1, rng.randint(1, per // 2)]))


def _sky(rng):
    J = rng.randint(8, 14)
    n_comp = _log(rng, 20, 50000)
    return dict(n_comp=n_comp, blobs=rng.choice([0, 20]), field=rng.choice([1.0, 2.0]), J=J), \
        max(20, min(n_comp, int(1700 * 3.0 ** (J - 12))))


def draw(rng):
    kind = rng.choice(["cycle", "cycle", "predict", "predict", "direct", "direct", "batched", "image", "clean",
                       "train", "truncated"])
    sign = rng.choice([1, -1])
    if kind in ("cycle", "predict"):
        sky, terms = _sky(rng)
        mode = rng.choice(["fp64", "df", "mixed", "fast", "tc"])
        if mode == "tc":
            sums = "eq16"
        elif mode == "df":
            sums = rng.choice(["regrouped", "eq16"])
        else:
            sums = rng.choice(["eq17", "regrouped", "eq16"])
        hi = min(4e6, 0.02 * RATES[mode] / terms)
        return dict(kind=kind, mode=mode, sum=sums, sign=sign, **sky, **_array(rng, hi))
    if kind == "direct":
        mode = rng.choice(["fp64", "df", "mixed", "fast", "tc"])
        n_comp = _log(rng, 20, 20000)
        hi = min(4e6, 0.02 * RATES[mode] / n_comp)
        return dict(kind=kind, mode=mode, sign=sign, n_comp=n_comp, blobs=rng.choice([0, 20]), field=2.0,
                    **_array(rng, hi, 300))
    if kind == "batched":
        n_ch = _log(rng, 2, 64)
        mode = rng.choice(["mixed", "fast"])
        hi = 0.02 * RATES[mode] / 2000 / n_ch
        return dict(kind=kind, n_ch=n_ch, n_comp=_log(rng, 500, 20000), blobs=20, field=2.0, J_lo=10,
                    J_hi=rng.randint(11, 13), mode=mode, sign=sign, **_array(rng, hi))
    if kind == "image":
        n = 2 * _log(rng, 128, 1024)
        planes = rng.choice([0, 0, 16, 32, 64, 128])
        a = _array(rng, 1.2e6)
        # the pixel that a program takes for its array: the longest baseline just inside the grid
        dl = 0.49 / (a["diameter"] * FREQ / C_LIGHT)
        if planes:          # the field, and with it the kernels, as wide as a 2048-pixel image of the medium array
            a["diameter"] = max(a["diameter"], 5000.0 * n / 2048)
            dl = min(0.49 / (a["diameter"] * FREQ / C_LIGHT), 0.043 / n)
        return dict(kind=kind, n=n, dl=dl, planes=planes, **a)
    if kind == "clean":
        return dict(kind=kind, n=2 * _log(rng, 32, 1024), iters=_log(rng, 50, 1500), gain=rng.choice([0.05, 0.1, 0.2]),
                    sources=rng.randint(10, 400))
    if kind == "train":
        return dict(kind=kind, samples=_log(rng, 20000, 2000000), batch=_log(rng, 1000, 32768),
                    steps=rng.randint(4, 32), lr=rng.choice([1e-3, 3e-3]), x_span=rng.uniform(6.0, 90.0))
    sky = dict(n_comp=_log(rng, 1000, 50000), blobs=20, field=2.0, J=rng.randint(11, 13))
    return dict(kind="truncated", level=sky["J"] - rng.randint(0, 2), sign=sign, **sky, **_array(rng, 3e6))


# ---------------------------------------------------------------- inputs

def _rng(seed, salt):
    return np.random.default_rng([int(seed) & 0xffffffff, salt])


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _uvw_metres(case, seed):
    """[n_vis, 3] metres, time-major, float64 on the GPU: hour angles over -1h .. +1h."""
    g = _rng(seed, 1)
    r = 0.5 * case["diameter"] * np.sqrt(g.random(case["n_ant"]))
    th = 2.0 * np.pi * g.random(case["n_ant"])
    e, nn = r * np.cos(th), r * np.sin(th)
    xyz = np.stack([-math.sin(LAT) * nn, e, math.cos(LAT) * nn], axis=1)
    i, j = np.triu_indices(case["n_ant"], k=1)
    X, Y, Z = (_dev((xyz[j] - xyz[i])[:, k]) for k in range(3))
    ha = _dev(np.linspace(-math.pi / 12, math.pi / 12, case["n_times"]) if case["n_times"] > 1 else np.array([0.1]))
    sh, ch = torch.sin(ha)[:, None], torch.cos(ha)[:, None]
    sd, cd = math.sin(DEC0), math.cos(DEC0)
    u = sh * X + ch * Y
    v = -sd * ch * X + sd * sh * Y + cd * Z
    w = cd * ch * X - cd * sh * Y + sd * Z
    out = torch.stack([u, v, w], dim=-1).reshape(-1, 3)
    return out[:out.shape[0] - case["drop"]].contiguous()


def _uvw(case, seed):
    return _uvw_metres(case, seed) * (FREQ / C_LIGHT)


def _components(case, seed, n_comp=None, salt=2):
    """(l, m, flux) as numpy arrays."""
    g = _rng(seed, salt)
    n = case["n_comp"] if n_comp is None else n_comp
    half = math.radians(case["field"]) / 2
    if case["blobs"]:
        c = g.uniform(-half, half, (2, case["blobs"]))
        at = g.integers(0, case["blobs"], n)
        lm = c[:, at] + math.radians(0.05) * g.standard_normal((2, n))
    else:
        lm = g.uniform(-half, half, (2, n))
    return lm[0], lm[1], 10.0 ** g.uniform(-3.0, 0.0, n)


def _channels(case, seed):
    """Per channel: frequency, J and component list of the batched workload."""
    g = _rng(seed, 3)
    freqs = np.linspace(1.0e9, 1.8e9, case["n_ch"])
    out = []
    for c in range(case["n_ch"]):
        n = int(round(10.0 ** g.uniform(2.0, math.log10(case["n_comp"]))))
        out.append((freqs[c], int(g.integers(case["J_lo"], case["J_hi"] + 1)), _components(case, seed, n, 100 + c)))
    return out


def _noise(shape, dtype, seed, scale=1.0):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7 + 5)
    return torch.randn(shape, dtype=dtype, device="cuda", generator=g) * scale


def _is_double(mode):
    return mode in ("fp64", "df")


def _net_params(seed, x_span):
    """Parameters of the scale a trained response network has: W1 [64][3], b1, W2 [64][64], b2, W3 [2][64], b3."""
    g = _rng(seed, 4)
    w1 = g.standard_normal((64, 3)) * (4.0 / x_span)
    b1 = g.standard_normal(64) * 0.5
    w2 = g.standard_normal((64, 64)) * math.sqrt(2.0 / 64)
    b2 = g.standard_normal(64) * 0.1
    w3 = g.standard_normal((2, 64)) * math.sqrt(1.0 / 64)
    b3 = np.array([0.3, 0.0])
    return np.concatenate([a.ravel() for a in (w1, b1, w2, b2, w3, b3)]).astype(np.float32)


def _train_data(case, seed):
    """Baselines (float64) whose |x| = |B| Delta theta reaches x_span, and a pixel-like response (float32 [n][2])."""
    level = 11
    scale = math.sqrt(math.pi / 3) * 2.0 ** (1 - level)
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 11 + 3)
    x = torch.rand((case["samples"], 3), dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    x = x * x.abs().amax(dim=1, keepdim=True) * case["x_span"]
    p, q = 0.7 * x[:, 0] + 0.2 * x[:, 1], -0.3 * x[:, 0] + 0.6 * x[:, 1] + 0.1 * x[:, 2]
    re = torch.sinc(p * 0.5) * torch.sinc(q * 0.5)
    im = 0.05 * torch.sin(0.1 * (p + q)) * torch.exp(-0.01 * (p * p + q * q))
    return level, x / scale, torch.stack([re, im], dim=1).to(torch.float32).contiguous()


def _clean_inputs(case, seed):
    """A dirty image and its beam, float32: point sources seen with an array's uv coverage (exact counts)."""
    n = case["n"]
    g = _rng(seed, 5)
    ant = (g.random((2, 40)) - 0.5) * 0.9 * (n // 2)
    i, j = np.triu_indices(40, k=1)
    b = ant[:, j] - ant[:, i]
    rot = np.linspace(-0.5, 0.5, 60)[:, None]
    iu = np.rint(np.cos(rot) * b[0] - np.sin(rot) * b[1]).astype(np.int64).ravel()
    iv = np.rint(0.7 * (np.sin(rot) * b[0] + np.cos(rot) * b[1])).astype(np.int64).ravel()
    grid = np.zeros((n, n))
    for s in (1, -1):
        np.add.at(grid, ((s * iv) % n, (s * iu) % n), 1.0)
    cov = _dev(grid / grid.sum())
    psf = torch.fft.fftshift(torch.fft.ifft2(cov).real) * (n * n)
    sky = np.zeros((n, n))
    span = max(2, int(0.35 * n))
    at = g.integers(n // 2 - span, n // 2 + span, (2, case["sources"]))
    np.add.at(sky, (at[0], at[1]), 10.0 ** g.uniform(-1.5, 0.3, case["sources"]))
    img = torch.fft.ifft2(torch.fft.fft2(_dev(sky)) * cov * (n * n)).real
    img = img + _noise((n, n), torch.float64, seed, 0.003)
    return img.to(torch.float32).contiguous(), psf.to(torch.float32).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("cycle", "predict", "direct", "truncated"):
        st["uvw"] = _uvw(case, seed)
        st["lmf"] = tuple(_dev(a) for a in _components(case, seed))
    if kind == "cycle":
        dt = torch.complex128 if _is_double(case["mode"]) else torch.complex64
        st["obs"] = _noise((st["uvw"].shape[0],), dt, seed, 5.0)
    if kind in ("predict", "truncated"):
        st["tree"] = wt.wt_build_tree(*st["lmf"], RA0, DEC0, case["J"])
    if kind == "truncated":
        span = case["diameter"] * FREQ / C_LIGHT * math.sqrt(math.pi / 3) * 2.0 ** (1 - case["level"])
        st["net"] = wt.Mlp(case["level"], RA0, DEC0, depth=3, x_max=1.001 * span, seed=1)
        st["net"].set_params(_net_params(seed, span))
    if kind == "batched":
        st["uvw_m"] = _uvw_metres(case, seed)
        ch = _channels(case, seed)
        st["freqs"] = [c[0] for c in ch]
        st["trees"] = [wt.wt_build_tree(*(_dev(a) for a in c[2]), RA0, DEC0, c[1]) for c in ch]
    if kind == "image":
        st["uvw"] = _uvw(case, seed)
        st["vis"] = _noise((st["uvw"].shape[0],), torch.complex64, seed) + 1.0
    if kind == "clean":
        st["image"], st["psf"] = _clean_inputs(case, seed)
    if kind == "train":
        level, st["x"], st["target"] = _train_data(case, seed)
        st["net"] = wt.Mlp(level, RA0, DEC0, depth=3, x_max=2 * case["x_span"], seed=1)
        st["params"] = _net_params(seed, case["x_span"])
    torch.cuda.synchronize()
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "cycle":
        mode = MODES[case["mode"]]
        tree = wt.wt_build_tree(*state["lmf"], RA0, DEC0, case["J"])
        vis = wt.wt_predict_vis(tree, state["uvw"], mode=mode, sign=case["sign"], which=SUMS[case["sum"]])
        resid = wt.subtract_model(state["obs"], vis, mode=mode)
        tree.close()
        return vis, resid
    if kind == "predict":
        return wt.wt_predict_vis(state["tree"], state["uvw"], mode=MODES[case["mode"]], sign=case["sign"],
                                 which=SUMS[case["sum"]])
    if kind == "direct":
        return wt.dft_predict_vis(*state["lmf"], state["uvw"], mode=MODES[case["mode"]], sign=case["sign"])
    if kind == "batched":
        return wt.wt_predict_vis_batched(state["trees"], state["freqs"], state["uvw_m"], mode=MODES[case["mode"]],
                                         sign=case["sign"])
    if kind == "image":
        if case["planes"]:
            return wt.wt_dirty_image_w(state["uvw"], state["vis"], case["n"], case["dl"], w_planes=case["planes"])
        return wt.wt_dirty_image(state["uvw"], state["vis"], case["n"], case["dl"])
    if kind == "clean":
        img = state["image"].clone()          # cleaned in place: the dirty image is kept
        pix, flux = wt.wt_hogbom(img, state["psf"], case["gain"], case["iters"])
        return img, pix, flux
    if kind == "train":
        net = state["net"]
        net.set_params(state["params"])
        loss = net.train(state["x"], state["target"], case["steps"], batch=case["batch"], lr=case["lr"])
        return loss, net.get_params()
    return wt.wt_predict_vis_truncated(state["tree"], case["level"], state["uvw"], response=wt.WT_RESPONSE_LEARNED,
                                       mlp=state["net"], sign=case["sign"])


# ---------------------------------------------------------------- the work a path cannot do without

def _n_vis(case):
    return case["n_ant"] * (case["n_ant"] - 1) // 2 * case["n_times"] - case["drop"]


def work(case):
    """Bytes: every input read once, every output written once. Operations of one term (a visibility against a leaf or
    component): three products and their sum for the phase, a sine, a cosine, two multiply-adds."""
    kind = case["kind"]
    term = 5 + 2 + 4
    if kind in ("cycle", "predict", "direct", "truncated"):
        n = _n_vis(case)
        out = 16 if _is_double(case.get("mode")) else 8
        b = n * (24 + out) + 24 * case["n_comp"]
        if kind == "direct":
            return dict(bytes=b, flops=n * case["n_comp"] * term)
        level = case.get("level", case["J"])
        leaves = len(np.unique(_keys(*_components(case, 1)[:2], level)))
        f = n * leaves * term
        if kind == "cycle":
            b += 2 * out * n                           # the data read, the residual written
            f += 2 * n
        if kind == "truncated":
            f += n * 2 * (3 * 64 + 64 * 64 + 2 * 64)
        return dict(bytes=b, flops=f)
    if kind == "batched":
        n = _n_vis(case)
        leaves = sum(len(np.unique(_keys(*c[2][:2], c[1]))) for c in _channels(case, 1))
        return dict(bytes=n * (24 + 8 * case["n_ch"]), flops=n * leaves * term)
    if kind == "image":
        n, nn = _n_vis(case), case["n"] ** 2
        fft = 5 * nn * math.log2(nn) / 2               # of a real image
        taps = 0
        if case["planes"]:
            taps = 9 * 9 * 8                           # the anti-aliasing kernel alone, interpolated between planes
        return dict(bytes=n * 32 + nn * 4, flops=n * max(4, taps) + fft)
    if kind == "clean":
        nn = case["n"] ** 2
        # every component touches what its beam overlaps: about three quarters of the image
        return dict(bytes=3 * 4 * nn + 8 * case["iters"], flops=2 * 0.75 * nn * case["iters"])
    per = 3 * 2 * (3 * 64 + 64 * 64 + 2 * 64)
    return dict(bytes=case["steps"] * case["batch"] * 32, flops=case["steps"] * case["batch"] * per)


# ---------------------------------------------------------------- the same in 64 bits, without the framework

def _rotation():
    """uvw -> xyz: R_y(ra0) R_x(-dec0) (Eq. 18)."""
    ca, sa, cd, sd = math.cos(RA0), math.sin(RA0), math.cos(-DEC0), math.sin(-DEC0)
    return np.array([[ca, sa * sd, sa * cd], [0.0, cd, -sd], [-sa, ca * sd, ca * cd]])


def _spread(x):
    out = np.zeros_like(x)
    for b in range(31):
        out |= ((x >> b) & 1) << (2 * b)
    return out


def _squeeze(x):
    out = np.zeros_like(x)
    for b in range(31):
        out |= ((x >> (2 * b)) & 1) << b
    return out


def _keys(l, m, J):
    """Nested pixel at level J (HEALPix order J - 1) of the image points (l, m)."""
    R = _rotation()
    n = np.sqrt(1.0 - (l * l + m * m))
    x, z, zc = (R[k, 0] * l + R[k, 1] * m + R[k, 2] * n for k in range(3))
    phi = np.arctan2(x, zc)
    phi = np.where(phi < 0, phi + 2 * np.pi, phi)
    order, ns = J - 1, 1 << (J - 1)
    t = phi / (0.5 * np.pi)
    a, b = ns * (0.5 + t), ns * (z * 0.75)
    up, dn = np.floor(a - b).astype(np.int64), np.floor(a + b).astype(np.int64)
    fu, fd = up >> order, dn >> order
    face = np.where(fu == fd, (fu & 3) + 4, np.where(fu < fd, fu, fd + 8))
    ix, iy = dn & (ns - 1), ns - 1 - (up & (ns - 1))
    q = np.minimum(t.astype(np.int64), 3)
    s = ns * np.sqrt(np.maximum(3.0 * (1.0 - np.abs(z)), 0.0))
    ja = np.minimum(np.floor((t - q) * s).astype(np.int64), ns - 1)
    jb = np.minimum(np.floor((1.0 - (t - q)) * s).astype(np.int64), ns - 1)
    cap, north = np.abs(z) > 2.0 / 3.0, z > 0
    face = np.where(cap, np.where(north, q, q + 8), face)
    ix = np.where(cap, np.where(north, ns - 1 - jb, ja), ix)
    iy = np.where(cap, np.where(north, ns - 1 - ja, jb), iy)
    return face * ns * ns + (_spread(ix) | (_spread(iy) << 1))


def _centres(keys, J):
    """(s_u, s_v, s_w - 1) of the pixels' centres."""
    order, ns = J - 1, 1 << (J - 1)
    face, inf = keys >> (2 * order), keys & (ns * ns - 1)
    ix, iy = _squeeze(inf), _squeeze(inf >> 1)
    row, col = face >> 2, face & 3
    ring = (row + 2) * ns - ix - iy - 1
    lon = np.where(row == 1, 2 * col, 2 * col + 1)
    north, south = ring < ns, ring > 3 * ns
    nr = np.where(north, ring, np.where(south, 4 * ns - ring, ns))
    d = nr.astype(np.float64) ** 2 / (3.0 * ns * ns)
    zb = (2 * ns - ring) * 2.0 / (3.0 * ns)
    z = np.where(north, 1.0 - d, np.where(south, d - 1.0, zb))
    st = np.where(north | south, np.sqrt(np.maximum(d * (2.0 - d), 0)), np.sqrt(np.maximum((1 - zb) * (1 + zb), 0)))
    shift = np.where(north | south, 0, (ring - ns) & 1)
    jp = (lon * nr + ix - iy + 1 + shift) // 2
    jp = np.where(jp > 4 * nr, jp - 4 * nr, jp)
    jp = np.where(jp < 1, jp + 4 * nr, jp)
    phi = (jp - 0.5 * (shift + 1)) * (0.5 * np.pi) / nr
    xyz = np.stack([st * np.sin(phi), z, st * np.cos(phi)], axis=1)
    s = xyz @ _rotation()                              # R^T xyz
    r2 = s[:, 0] ** 2 + s[:, 1] ** 2
    return np.stack([s[:, 0], s[:, 1], np.where(s[:, 2] > 0, -r2 / (1.0 + s[:, 2]), s[:, 2] - 1.0)], axis=1)


def _pixels(l, m, flux, J):
    """The occupied level-J pixels' centres and merged fluxes."""
    keys, at = np.unique(_keys(l, m, J), return_inverse=True)
    return _centres(keys, J), np.bincount(at.ravel(), weights=flux, minlength=len(keys))


def _plane_waves(uvw, dirs, flux, sign):
    """sum_k flux_k exp(sign i 2 pi B . d_k) in float64, blocks of visibilities at a time."""
    D, F = _dev(dirs).T.contiguous(), _dev(flux)
    n = uvw.shape[0]
    out = torch.empty(n, dtype=torch.complex128, device="cuda")
    step = max(1, int(4e7 // max(1, D.shape[1])))
    for a in range(0, n, step):
        b = uvw[a:a + step]
        t = b[:, :1] * D[0] + b[:, 1:2] * D[1] + b[:, 2:] * D[2]
        t -= torch.round(t)
        t *= sign * 2 * math.pi
        out[a:a + step] = torch.complex(torch.cos(t) @ F, torch.sin(t) @ F)
    return out


def _network(params, x):
    """The 3 -> 64 -> 64 -> 2 network in float64, W2 and the first hidden layer rounded to bfloat16 as documented."""
    w1, b1, w2, b2, w3, b3 = _unpack(params)
    silu = torch.nn.functional.silu
    h = silu(x @ w1.T + b1).to(torch.bfloat16).to(torch.float64)
    return silu(h @ w2.to(torch.bfloat16).to(torch.float64).T + b2) @ w3.T + b3


def _unpack(p):
    out, at = [], 0
    for shape in ((64, 3), (64,), (64, 64), (64,), (2, 64), (2,)):
        n = int(np.prod(shape))
        out.append(p[at:at + n].reshape(shape))
        at += n
    return out


def _exact_image(case, seed):
    n, dl = case["n"], case["dl"]
    uvw = _uvw(case, seed)
    vis = (_noise((uvw.shape[0],), torch.complex64, seed) + 1.0).to(torch.complex128)
    grid = torch.zeros(n * n, dtype=torch.complex128, device="cuda")
    half = n // 2
    x, y, w = uvw[:, 0] * (n * dl), uvw[:, 1] * (n * dl), uvw[:, 2]
    ic, jc = torch.round(x), torch.round(y)
    k = torch.arange(n, device="cuda", dtype=torch.float64) - half
    if not case["planes"]:
        ok = (ic.abs() < half) & (jc.abs() < half)
        at = ((jc[ok].long() % n) * n + ic[ok].long() % n)
        grid.index_put_((at,), vis[ok], accumulate=True)
        entries, taper = int(ok.sum()), torch.ones(n, dtype=torch.float64, device="cuda")
    else:
        width, beta, over, M, P = 7, 16.25, 8, 128, case["planes"]

        def kb(t):
            a = beta * beta - (math.pi * width * t) ** 2
            r = torch.sqrt(a.abs())
            return torch.where(a > 0, torch.sinh(r), torch.sin(r)) / r / (math.sinh(beta) / beta)

        w_max = float(w.abs().max()) or 1.0
        ndl = n * dl
        per_w = ndl * ndl / (2.0 * math.sqrt(1.0 - 0.5 * ndl * ndl))
        h = int(math.ceil(0.5 * width + w_max * per_w)) + 1
        T, dw = (2 * h + 1) * over + 1, w_max / (P - 1)
        t = (torch.arange(M, device="cuda", dtype=torch.float64) + 0.5) / M - 0.5
        r2 = (t * ndl)[:, None] ** 2 + (t * ndl)[None, :] ** 2
        nm1 = -r2 / (1.0 + torch.sqrt(1.0 - r2))
        c2 = kb(t)[:, None] * kb(t)[None, :]
        xs = torch.arange(T, device="cuda", dtype=torch.float64) / over - (h + 0.5)
        tw = torch.exp(2j * math.pi * (xs[:, None] * t[None, :]))
        K = torch.empty((P + 1, T, T), dtype=torch.complex128, device="cuda")
        for p in range(P):
            K[p] = tw @ (c2 * torch.exp(-2j * math.pi * (p * dw) * nm1)) @ tw.T / (M * M)
        K[P] = 0
        lim = half - h - 1
        ok = (ic >= -lim) & (ic <= lim) & (jc >= -lim) & (jc <= lim)
        entries = int(ok.sum())
        x, y, w, vis, ic, jc = x[ok], y[ok], w[ok], vis[ok], ic[ok], jc[ok]
        pw = w.abs() / dw
        p0 = pw.floor().long().clamp(0, P - 2)
        a = (pw - p0).clamp(0, 1)
        he = torch.minimum(torch.ceil(0.5 * width + per_w * w.abs()).long() + 1, torch.tensor(h, device="cuda"))
        neg = w < 0
        # the table's nearest offset as single precision finds it (the documented 8 points per cell)
        fx, fy = (x - ic).float(), (y - jc).float()
        for dy in range(-h, h + 1):
            for dx in range(-h, h + 1):
                on = (he >= max(abs(dx), abs(dy))).nonzero().squeeze(1)
                if not on.numel():
                    continue
                s = neg[on]
                ix = torch.round((dx - fx[on] + (h + 0.5)) * over).long().clamp(0, T - 1)
                iy = torch.round((dy - fy[on] + (h + 0.5)) * over).long().clamp(0, T - 1)
                ix, iy = torch.where(s, T - 1 - ix, ix), torch.where(s, T - 1 - iy, iy)
                k0, k1 = K[p0[on], ix, iy], K[p0[on] + 1, ix, iy]
                kk = k0 + a[on] * (k1 - k0)
                kk = torch.where(s, kk.conj(), kk)
                at = ((jc[on].long() + dy) % n) * n + (ic[on].long() + dx) % n
                grid.index_put_((at,), vis[on] * kk, accumulate=True)
        taper = kb(k / n)
    # the entries and their conjugates at the mirrored cells: twice the real part of the transform
    img = torch.fft.fftshift(torch.fft.fft2(grid.reshape(n, n))).real / max(1, entries)
    return img / (taper[:, None] * taper[None, :])


def _exact_train(case, seed):
    level, uvw, target = _train_data(case, seed)
    scale = math.sqrt(math.pi / 3) * 2.0 ** (1 - level)
    x, target = uvw * scale, target.to(torch.float64)
    p = _dev(_net_params(seed, case["x_span"])).to(torch.float64)
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    n, first, loss = case["samples"], 0, 0.0

    def rounded(z):                                    # to bfloat16, the gradient passed through
        return z + (z.detach().to(torch.bfloat16).to(torch.float64) - z.detach())

    silu = torch.nn.functional.silu
    for it in range(case["steps"]):
        at = (first + torch.arange(case["batch"], device="cuda")) % n
        q = p.clone().requires_grad_(True)
        w1, b1, w2, b2, w3, b3 = _unpack(q)
        h = rounded(silu(x[at] @ w1.T + b1))
        y = silu(h @ rounded(w2).T + b2) @ w3.T + b3
        e = ((y - target[at]) ** 2).sum() / case["batch"]
        g, = torch.autograd.grad(e, q)
        loss = float(e)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        lr = 0.5 * case["lr"] * (1.0 + math.cos(math.pi * it / case["steps"]))
        p = p - lr * (m / (1 - 0.9 ** (it + 1))) / (torch.sqrt(v / (1 - 0.999 ** (it + 1))) + 1e-8)
        first = (first + case["batch"]) % n
    return loss, p.cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("cycle", "predict", "direct", "truncated"):
        uvw, (l, m, f) = _uvw(case, seed), _components(case, seed)
        if kind == "direct":
            r2 = l * l + m * m
            return _plane_waves(uvw, np.stack([l, m, -r2 / (1.0 + np.sqrt(1.0 - r2))], axis=1), f, case["sign"])
        vis = _plane_waves(uvw, *_pixels(l, m, f, case.get("level", case["J"])), case["sign"])
        if kind == "predict":
            return vis
        if kind == "cycle":
            dt = torch.complex128 if _is_double(case["mode"]) else torch.complex64
            return vis, _noise((uvw.shape[0],), dt, seed, 5.0).to(torch.complex128) - vis
        scale = math.sqrt(math.pi / 3) * 2.0 ** (1 - case["level"])
        p = _dev(_net_params(seed, case["diameter"] * FREQ / C_LIGHT * scale)).to(torch.float64)
        for a in range(0, uvw.shape[0], 1 << 20):
            y = _network(p, uvw[a:a + (1 << 20)] * scale)
            vis[a:a + (1 << 20)] *= torch.complex(y[:, 0], case["sign"] * y[:, 1])
        return vis
    if kind == "batched":
        uvw_m = _uvw_metres(case, seed)
        return torch.stack([_plane_waves(uvw_m * (f / C_LIGHT), *_pixels(*lmf, J), case["sign"])
                            for f, J, lmf in _channels(case, seed)])
    if kind == "image":
        return _exact_image(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    return None                                        # clean: a chain of decisions in single precision
