"""The work a user has this library do, as measurable cases.

Each case is one call, or the few calls that belong together, through the
public entry points (the binding of the C ABI, ``autotune``, ``estimator``),
on inputs a program has in hand: stacks of blob specimens imaged with the
optics of the case plus 1e-3 noise, and the banks, workspaces and weights such
a program keeps.  ``exact`` restates the outputs in plain float64 torch.

The families and what they stand for:

recon     Tikhonov reconstruction with a bank built beforehand, 3D or 2D
shared    a batch of stacks of one microscope sharing one bank
tf        the transfer-function build from host optics
model     the forward model and its adjoint, as an iterative solver calls them
field     a shift-variant field: bank from device optics, tiles, blend
tune      one evaluation of the auto-tuning loss and gradient
fused     several illumination apertures fused into one phase volume
train     loss and weight gradients of the estimator's network
predict   spectra, features and network outputs of a batch of tiles
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2412_09775_gb300 import autotune as A
from paper_2412_09775_gb300 import binding as B
from paper_2412_09775_gb300 import estimator as E

DEV = "cuda"
ETA = 1e-3
OPTICS = dict(lambda_um=0.532, n_medium=1.33, pixel_um=0.1, z_step_um=0.25, na_det=1.2, na_ill=0.9,
              tilt_x=0.0, tilt_y=0.0, defocus_um=0.0)
SCREEN_OPTICS = dict(lambda_um=0.45, n_medium=1.0, pixel_um=0.65, z_step_um=2.0, na_det=0.15, na_ill=0.1,
                     tilt_x=0.0, tilt_y=0.0, defocus_um=0.0)
LAYERS = ((3, 32, 1), (32, 64, 2), (64, 96, 2), (96, 128, 2))  # in, out, stride of the estimator's convolutions


# --------------------------------------------------------------------- cases
def listed():
    return [
        # one small brightfield z-stack of a pooled screen: latency and launches count
        dict(name="stack_16x64x64", op="recon", n=1, Z=16, Y=64, X=64, kinds="phase", mode="3d", optics="oil"),
        # the screen's whole batch of such stacks, one microscope, one bank
        dict(name="stacks_4096x16x64x64", op="shared", n=4096, Z=16, Y=64, X=64, kinds="phase", kx_major=True,
             optics="oil"),
        # the joint widefield volume: build its bank, then reconstruct with a bank at hand
        dict(name="widefield_tf_96x512x512", op="tf", n=1, Z=96, Y=512, X=512, kinds="phase+absorption+fluor",
             optics="oil"),
        dict(name="widefield_recon_96x512x512", op="recon", n=1, Z=96, Y=512, X=512,
             kinds="phase+absorption+fluor", mode="3d", optics="oil"),
        # the forward model and its adjoint on oblong volumes of an iterative solver, each with its own optics
        dict(name="model_2x24x384x768", op="model", n=2, Z=24, Y=384, X=768, kinds="phase+fluor", optics="tiles"),
        # the shift-variant field: 256 tiles of 48x192x192, each with its own optics
        dict(name="field_48x2048x2048", op="field", Z=48, tiles_y=16, tiles_x=16, core=128, halo=32, kinds="phase",
             kx_major=True, optics="tiles"),
        # 2D phase from defocus of a pooled screen's 6 x 6 tiles
        dict(name="screen2d_36x24x256x256", op="recon", n=36, Z=24, Y=256, X=256, kinds="phase", mode="2d",
             optics="screen"),
        # one auto-tuning evaluation of the field's tiles in all four parameters
        dict(name="tune4_256x48x192x192", op="tune", n=256, Z=48, Y=192, X=192, params="all", optics="tiles"),
        # and of the screen's tiles in their defocus alone
        dict(name="tune1_36x24x256x256", op="tune", n=36, Z=24, Y=256, X=256, params="defocus", optics="screen"),
        # nine illumination apertures (one on axis, eight on a ring) fused per tile
        dict(name="fused_4x9x32x128x128", op="fused", n=4, channels=9, Z=32, Y=128, X=128, mode="3d"),
        # the estimator: a training batch's gradients, and a batch of tiles from stack to predicted optics
        dict(name="estimator_train_256", op="train", n=256),
        dict(name="estimator_predict_256x48x128x128", op="predict", n=256, Z=48, Y=128, X=128, optics="tiles"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, zs, ys, xs, lo, hi):
    """Z, Y, X from the lists and a tile count, n Z Y X log-uniform in [lo, hi]."""
    Z, Y, X = rng.choice(zs), rng.choice(ys), rng.choice(xs)
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    while Z * Y * X > hi:
        Z, Y, X = rng.choice(zs), rng.choice(ys), rng.choice(xs)
    return max(1, min(int(want / (Z * Y * X)), 2048)), Z, Y, X


def draw(rng):
    zs, lat = (6, 8, 12, 16, 24, 32, 48, 64, 96), (48, 64, 96, 128, 192, 256, 384, 512, 768)
    kinds = ("phase", "absorption", "fluor", "phase+absorption", "phase+fluor", "phase+absorption+fluor")
    op = rng.choice(("recon", "shared", "tf", "model", "field", "tune", "tune", "fused", "train", "predict", "recon"))
    if op == "recon":
        mode = rng.choice(("3d", "3d", "2d"))
        n, Z, Y, X = _size(rng, zs, lat, lat, 6e4, 2.6e7)
        k = rng.choice(kinds)
        optics = rng.choice(("oil", "tiles", "screen") if k == "phase" else ("oil", "tiles"))
        return dict(op=op, n=n, Z=Z, Y=Y, X=X, kinds=k, mode=mode, optics=optics)
    if op == "shared":
        if rng.random() < 0.5:
            Z, E_ = rng.choice(((16, 64), (32, 64), (48, 128), (32, 128), (48, 192)))
            n = max(1, int(math.exp(rng.uniform(math.log(2e5), math.log(2.6e8))) / (Z * E_ * E_)))
            return dict(op=op, n=n, Z=Z, Y=E_, X=E_, kinds="phase", kx_major=True, optics="oil")
        n, Z, Y, X = _size(rng, (6, 12, 16, 24), (48, 64, 96, 128), (48, 64, 96, 128), 2e5, 1e8)
        return dict(op=op, n=n, Z=Z, Y=Y, X=X, kinds=rng.choice(kinds[:2]), kx_major=False, optics="oil")
    if op == "tf":
        n, Z, Y, X = _size(rng, zs, lat, lat, 6e4, 2.6e7)
        return dict(op=op, n=n, Z=Z, Y=Y, X=X, kinds=rng.choice(kinds), optics=rng.choice(("oil", "tiles")))
    if op == "model":
        n, Z, Y, X = _size(rng, zs, lat, lat, 6e4, 2.6e7)
        return dict(op=op, n=n, Z=Z, Y=Y, X=X, kinds=rng.choice(kinds), optics=rng.choice(("oil", "tiles")))
    if op == "field":
        Z, core, halo, kxm = rng.choice(((48, 128, 32, True), (32, 128, 32, True), (48, 96, 16, True),
                                         (32, 48, 8, True), (16, 48, 8, True), (24, 64, 16, False),
                                         (48, 128, 32, False), (12, 144, 24, False), (24, 192, 32, False)))
        k = rng.choice(("phase", "absorption", "fluor") if kxm else ("phase", "fluor", "phase+absorption"))
        return dict(op=op, Z=Z, tiles_y=_log_int(rng, 1, 13), tiles_x=_log_int(rng, 1, 13), core=core, halo=halo,
                    kinds=k, kx_major=kxm, optics="tiles")
    if op == "tune":
        if rng.random() < 0.5:
            n, Z, Y, X = _size(rng, (8, 12, 16, 24, 32, 48), (48, 64, 96, 128, 192, 256),
                               (48, 64, 96, 128, 192, 256), 2e5, 3e8)
            return dict(op=op, n=min(n, 256), Z=Z, Y=Y, X=X, params="all", optics="tiles")
        n, Z, Y, X = _size(rng, (6, 8, 12, 16, 24, 32), (64, 96, 128, 192, 256, 384), (64, 96, 128, 192, 256, 384),
                           2e5, 1e8)
        return dict(op=op, n=min(n, 256), Z=Z, Y=Y, X=X, params="defocus", optics=rng.choice(("screen", "tiles")))
    if op == "fused":
        Z, Y, X = rng.choice((12, 16, 24, 32, 48)), rng.choice((48, 64, 96, 128)), rng.choice((48, 64, 96, 128))
        c = rng.randint(2, 9)
        n = max(1, int(math.exp(rng.uniform(math.log(2e5), math.log(2e7))) / (c * Z * Y * X)))
        return dict(op=op, n=n, channels=c, Z=Z, Y=Y, X=X, mode=rng.choice(("3d", "2d")))
    if op == "train":
        return dict(op=op, n=_log_int(rng, 8, 256))
    Z, Y, X = rng.choice(((16, 64, 64), (24, 96, 128), (48, 128, 128), (32, 192, 192)))
    return dict(op="predict", n=min(256, max(1, int(2e8 / (Z * Y * X) * rng.random()))), Z=Z, Y=Y, X=X,
                optics="tiles")


# ------------------------------------------------------- optics and specimens
def _kinds(case):
    return tuple(case["kinds"].split("+"))


def _mask(case):
    return B.kinds_mask(_kinds(case)) | (B.WO_TF_KX_MAJOR if case.get("kx_major") else 0)


def _shape(case):
    if case["op"] == "field":
        e = case["core"] + 2 * case["halo"]
        return case["tiles_y"] * case["tiles_x"], case["Z"], e, e
    return case["n"], case["Z"], case["Y"], case["X"]


def _optics(case, seed, n=None):
    """The true optics of every tile."""
    rng = np.random.default_rng(seed)
    n = case["n"] if n is None else n
    base = SCREEN_OPTICS if case["optics"] == "screen" else OPTICS
    if case["optics"] == "oil":  # one objective, a small focus error
        return [dict(base, defocus_um=float(rng.uniform(-0.2, 0.2)))] * n
    out = []
    for _ in range(n):
        if case["optics"] == "screen":
            out.append(dict(base, defocus_um=float(rng.uniform(-4, 4)), tilt_x=float(rng.uniform(-0.02, 0.02)),
                            tilt_y=float(rng.uniform(-0.02, 0.02))))
        else:
            out.append(dict(base, defocus_um=float(rng.uniform(-1, 1)), tilt_x=float(rng.uniform(-0.1, 0.1)),
                            tilt_y=float(rng.uniform(-0.1, 0.1)), na_ill=float(rng.uniform(0.7, 0.95))))
    return out


def _start_optics(case, true):
    """Where tuning starts: nominal optics (the screen keeps its known illumination)."""
    if case["params"] == "all":
        return [dict(o, defocus_um=0.0, tilt_x=0.0, tilt_y=0.0, na_ill=0.825) for o in true]
    return [dict(o, defocus_um=0.0) for o in true]


def _apertures(case, seed):
    """One aperture on axis and the others on a ring of 0.6 NA, each of 0.15 NA, per tile with its own defocus."""
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(case["n"]):
        z0, c = float(rng.uniform(-0.3, 0.3)), case["channels"]
        for i in range(c):
            a = 2.0 * math.pi * (i - 1) / max(c - 1, 1)
            r = 0.0 if i == 0 else 0.6
            out.append(dict(OPTICS, na_ill=0.15, tilt_x=r * math.cos(a), tilt_y=r * math.sin(a), defocus_um=z0))
    return out


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _blobs(shape, pitch, gen):
    """Blobs about a micrometre (ten in low-NA screens) across, values up to 0.02, on the last len(pitch) axes."""
    d = len(pitch)
    dims = tuple(range(-d, 0))
    size = 0.5 if pitch[-1] < 0.3 else 3.0
    v = torch.fft.rfftn(torch.randn(shape, generator=gen, device=DEV), dim=dims)
    for i, p in zip(dims, pitch):
        n = shape[i]
        k = torch.arange(v.shape[i], device=DEV, dtype=torch.float32)
        k = torch.where(k < (n + 1) // 2 + 1, k, k - n) / (n * p)
        v *= torch.exp(-2.0 * (math.pi * size * k) ** 2).reshape([-1] + [1] * (-1 - i))
    v = torch.fft.irfftn(v, s=[shape[i] for i in dims], dim=dims)
    v /= v.std().clamp_min(1e-20)
    return 0.02 * torch.sigmoid(6.0 * (v - 1.0))


# ------------------------------------------------- transfer functions in torch
def _axis(n, p):
    k = torch.arange(n, device=DEV, dtype=torch.float64)
    return torch.where(k < (n + 1) // 2, k, k - n) / (float(n) * p)


def _plane_tfs(o, Z, Y, X, kinds, real=torch.float64, theta=None, smooth=False):
    """Per-plane half spectra {kind: [Z, Y, X/2+1]} of the scalar weak-object transfer functions; theta
    (defocus, tilt_x, tilt_y, na_ill as float64 tensors) takes the place of the optics' own."""
    lam, km = o["lambda_um"], o["n_medium"] / o["lambda_um"]
    z0, tx, ty, na = theta if theta is not None else (o["defocus_um"], o["tilt_x"], o["tilt_y"], o["na_ill"])
    ny, nx = _axis(Y, o["pixel_um"])[:, None], _axis(X, o["pixel_um"])[None, :]
    r2 = nx * nx + ny * ny
    rp = o["na_det"] / lam
    P = (r2 <= rp * rp).to(torch.float64)
    eta = torch.sqrt(torch.clamp(km * km - r2, min=0.0))
    j = torch.arange(Z, device=DEV, dtype=torch.float64)
    z = torch.where(j < (Z + 1) // 2, j, j - Z) * o["z_step_um"] + z0
    cyc = eta[None] * z[:, None, None]
    ph = 2.0 * math.pi * (cyc - torch.round(cyc.detach())).to(real)
    prop = torch.complex(torch.cos(ph), torch.sin(ph)) * P.to(real)
    out, N = {}, Y * X
    if "phase" in kinds or "absorption" in kinds:
        dx, dy = nx - tx / lam, ny - ty / lam
        d2 = dx * dx + dy * dy
        if smooth:
            w = 1.0 / (min(Y, X) * o["pixel_um"])
            d = torch.sqrt(torch.where(d2 > 0, d2, torch.ones_like(d2))) * (d2 > 0)
            S = 1.0 / (1.0 + torch.exp(-(na / lam - d) / w))
        else:
            rs = na / lam
            S = (d2 <= rs * rs).to(torch.float64)
        norm = torch.sum(S * P)
        a = torch.fft.ifft2(S.to(real) * prop)
        b = torch.fft.ifft2(torch.where(P > 0, 1.0 / torch.where(P > 0, eta, torch.ones_like(eta)),
                                        torch.zeros_like(eta)).to(real) * prop * 1j)
        g = torch.conj(a) * b
        c = 2.0 * math.pi * o["n_medium"] * o["z_step_um"] / lam ** 2
        K = (2.0 * c * N / norm).to(real)
        if "phase" in kinds:
            out["phase"] = torch.fft.rfft2(K * g.real)
        if "absorption" in kinds:
            out["absorption"] = torch.fft.rfft2(-K * g.imag)
    if "fluor" in kinds:
        p = torch.fft.ifft2(prop)
        out["fluor"] = torch.fft.rfft2((p.real ** 2 + p.imag ** 2) * (N / (Z * torch.sum(P))).to(real))
    return out


def _tfs(o, Z, Y, X, kinds, real=torch.float64, smooth=False):
    return {k: torch.fft.fft(v, dim=0) for k, v in _plane_tfs(o, Z, Y, X, kinds, real, smooth=smooth).items()}


def _modes(kinds):
    """The contrast modes: (channel, its properties as (index, kind)); label-free first."""
    props = [k for k in ("phase", "absorption", "fluor") if k in kinds]
    lf = [(props.index(k), k) for k in props if k != "fluor"]
    out = [(0, lf)] if lf else []
    if "fluor" in kinds:
        out.append((len(out), [(props.index("fluor"), "fluor")]))
    return out, len(props)


def _each(optics):
    """Runs of tiles with the same optics: (optics, first, end)."""
    i = 0
    while i < len(optics):
        j = i + 1
        while j < len(optics) and optics[j] == optics[i]:
            j += 1
        yield optics[i], i, j
        i = j


def _chunks(lo, hi, size):
    for i in range(lo, hi, size):
        yield i, min(i + size, hi)


def _specimen(n, kinds, Z, Y, X, o, gen):
    """Properties [n, P, Z, Y, X] (float32): index increment, extinction, fluorophore density."""
    scale = {"phase": 1.0, "absorption": 0.3, "fluor": 50.0}
    P = [k for k in ("phase", "absorption", "fluor") if k in kinds]
    f = torch.empty((n, len(P), Z, Y, X), device=DEV)
    for lo, hi in _chunks(0, n, max(1, 64000000 // (Z * Y * X))):
        for i, k in enumerate(P):
            f[lo:hi, i] = scale[k] * _blobs((hi - lo, Z, Y, X), (o["z_step_um"], o["pixel_um"], o["pixel_um"]), gen)
    return f


def _image(H, f, kinds):
    """Data [n, C, Z, Y, X] of properties f through the half-spectrum TFs H, background 1."""
    modes, _ = _modes(kinds)
    d = []
    for _, ps in modes:
        s = sum(H[k] * torch.fft.rfftn(f[:, i], dim=(-3, -2, -1)) for i, k in ps)
        d.append(torch.fft.irfftn(s, s=f.shape[-3:], dim=(-3, -2, -1)) + 1.0)
    return torch.stack(d, dim=1)


def _stacks(case, optics, gen):
    """Data [n, C, Z, Y, X] (float32) of 3D specimens with every tile's optics."""
    n, Z, Y, X = _shape(case)
    kinds = _kinds(case)
    modes, _ = _modes(kinds)
    d = torch.empty((n, len(modes), Z, Y, X), device=DEV)
    for o, i, j in _each(optics):
        H = _tfs(o, Z, Y, X, kinds, torch.float32)
        for lo, hi in _chunks(i, j, max(1, 32000000 // (Z * Y * X))):
            d[lo:hi] = _image(H, _specimen(hi - lo, kinds, Z, Y, X, o, gen), kinds)
    return _add_noise(d, gen)


def _thin_stacks(optics, Z, Y, X, gen, smooth=False):
    """Data [n, Z, Y, X] of thin specimens: plane j sees the per-plane TF H_j."""
    n = len(optics)
    f = 5.0 * _blobs((n, Y, X), (optics[0]["pixel_um"],) * 2, gen)
    d = torch.empty((n, Z, Y, X), device=DEV)
    for t, o in enumerate(optics):
        H = _plane_tfs(o, Z, Y, X, ("phase",), torch.float32, smooth=smooth)["phase"]
        d[t] = torch.fft.irfft2(H * torch.fft.rfft2(f[t]), s=(Y, X)) + 1.0
    return _add_noise(d, gen)


def _add_noise(d, gen):
    for lo, hi in _chunks(0, d.shape[0], max(1, 64000000 // max(d[0].numel(), 1))):
        d[lo:hi] += 1e-3 * torch.randn(d[lo:hi].shape, generator=gen, device=DEV)
    return d


def _window(start, size, n, mirror):
    i = torch.arange(start, start + size, device=DEV)
    if not mirror:
        return i % n
    i = torch.where(i < 0, -i, i)
    return torch.where(i >= n, 2 * (n - 1) - i, i)


def _field(case, optics, gen):
    """A field whose cores are imaged with each tile's own optics."""
    n, Z, e, _ = _shape(case)
    kinds, core, halo = _kinds(case), case["core"], case["halo"]
    Yf, Xf = case["tiles_y"] * core, case["tiles_x"] * core
    f = _specimen(1, kinds, Z, Yf, Xf, optics[0], gen)
    out = torch.empty((1, Z, Yf, Xf), device=DEV)
    for t, o in enumerate(optics):
        y0, x0 = t // case["tiles_x"] * core, t % case["tiles_x"] * core
        ys, xs = _window(y0 - halo, e, Yf, False), _window(x0 - halo, e, Xf, False)
        d = _image(_tfs(o, Z, e, e, kinds, torch.float32), f[:, :, :, ys][..., xs], kinds)
        out[:, :, y0:y0 + core, x0:x0 + core] = d[0, :, :, halo:halo + core, halo:halo + core]
    return _add_noise(out, gen)[0]


# ------------------------------------------------------------------- estimator
def _weights(seed):
    """A flat parameter array of a network on its way through training (He-normal weights, small biases)."""
    rng = np.random.default_rng(seed)
    parts = []
    for ci, co, _ in LAYERS:
        parts += [rng.normal(0.0, math.sqrt(2.0 / (9 * ci)), co * ci * 9), rng.normal(0.0, 0.02, co)]
    parts += [rng.normal(0.0, math.sqrt(1.0 / 128), 4 * 128), rng.normal(0.0, 0.02, 4)]
    return torch.from_numpy(np.concatenate(parts).astype(np.float32)).to(DEV)


def _features(n, gen):
    """Feature images with the values wo_est_features gives: a power profile peaked in the focal planes and at
    low frequencies, drifts in [-1, 1], 48 of the 64 plane rows filled."""
    row = torch.arange(64, device=DEV, dtype=torch.float32)[:, None]
    col = torch.arange(64, device=DEV, dtype=torch.float32)[None, :]
    focus = 24.0 + 8.0 * (torch.rand((n, 1, 1), generator=gen, device=DEV) - 0.5)
    power = torch.exp(-col / 8.0) * (1.0 + 20.0 * torch.exp(-((row - focus) / (3.0 + col / 8.0)) ** 2))
    noise = torch.rand((n, 3, 64, 64), generator=gen, device=DEV)
    f = torch.empty((n, 3, 64, 64), device=DEV)
    f[:, 0] = torch.log1p(8.0 * power * (0.5 + noise[:, 0]))
    drift = torch.rand((n, 2, 1, 1), generator=gen, device=DEV) - 0.5
    f[:, 1:] = drift * torch.sin(col / 10.0) + 0.2 * (noise[:, 1:] - 0.5)
    f[:, :, 48:] = 0.0
    return f


def _targets(n, seed):
    rng = np.random.default_rng(seed)
    t = np.stack([rng.uniform(-1, 1, n), rng.uniform(-0.1, 0.1, n), rng.uniform(-0.1, 0.1, n),
                  rng.uniform(0.7, 0.95, n)], axis=1)
    return torch.from_numpy(t.astype(np.float32)).to(DEV)


def _network64(w, feat, grad=False):
    """The network in float64 (weights rounded to bfloat16): outputs and, for grad, its parameters."""
    params, i, h = [], 0, feat.to(torch.float64)

    def take(*shape, rounded):
        nonlocal i
        k = math.prod(shape)
        v = w[i:i + k].reshape(shape)
        i += k
        v = (v.to(torch.bfloat16) if rounded else v).to(torch.float64).requires_grad_(grad)
        params.append(v)
        return v

    for ci, co, s in LAYERS:
        k, bias = take(co, ci, 3, 3, rounded=True), take(co, rounded=False)
        h = torch.relu(torch.nn.functional.conv2d(h, k, bias, stride=s, padding=1))
    lin, bias = take(4, 128, rounded=True), take(4, rounded=False)
    return h.mean(dim=(2, 3)) @ lin.T + bias, params


# ------------------------------------------------------------- prepare and run
def prepare(case, seed):
    op, gen = case["op"], _gen(seed)
    st = dict(case=case)
    if op == "train":
        n = case["n"]
        w = _weights(seed)
        st.update(w=w, wbf=torch.empty(w.numel(), dtype=torch.int16, device=DEV), feat=_features(n, gen),
                  target=_targets(n, seed + 1), grad=torch.empty_like(w), loss=torch.zeros(1, device=DEV),
                  ws=torch.empty(B.wo_est_workspace_bytes(n), dtype=torch.uint8, device=DEV))
        B.wo_est_sync_bf16(st["w"], st["wbf"])
        return st
    if op == "fused":
        n, C, Z, Y, X = case["n"], case["channels"], case["Z"], case["Y"], case["X"]
        ol = _apertures(case, seed)
        f = _specimen(n, ("phase",), Z, Y, X, OPTICS, gen)
        d = torch.empty((n, C, Z, Y, X), device=DEV)
        for t in range(n):
            for c in range(C):
                d[t, c] = _image(_tfs(ol[t * C + c], Z, Y, X, ("phase",), torch.float32), f[t:t + 1],
                                 ("phase",))[0, 0]
        tf, ws0 = B.alloc(n * C, Z, Y, X, "phase", DEV)
        B.wo_build_tf(ol, n * C, Z, Y, X, "phase", tf, ws0)
        ws = torch.zeros(B.wo_fused_workspace_bytes(C, n, Z, Y, X), dtype=torch.uint8, device=DEV)
        out = torch.empty((n, Z, Y, X) if case["mode"] == "3d" else (n, Y, X), device=DEV)
        st.update(data=_add_noise(d, gen), tf=tf, ws=ws, out=out)
        return st
    n, Z, Y, X = _shape(case)
    ol = _optics(case, seed, n)
    if op == "tune":
        data = _thin_stacks(ol, Z, Y, X, gen, smooth=case["params"] == "all")
        st["problem"] = A.TuningProblem(data, _start_optics(case, ol), ETA, params=case["params"])
        return st
    if op == "predict":
        est = E.Estimator(torch.device(DEV), batch=min(n, 256))
        est.w32.copy_(_weights(seed))
        B.wo_est_sync_bf16(est.w32, est.wbf)
        st.update(est=est, data=_thin_stacks(ol, Z, Y, X, gen, smooth=True), optics=B.optics_tensor(ol, DEV),
                  spec=torch.empty((n, Z, Y, X // 2 + 1), dtype=torch.complex64, device=DEV),
                  feat=torch.empty((n, 3, 64, 64), device=DEV))
        return st
    kinds, mask = _kinds(case), _mask(case)
    modes, P = _modes(kinds)
    st.update(kinds=mask, eta=[ETA] * len(modes))
    if op == "field":
        st["field"] = _field(case, ol, gen)
        st["optics"] = B.optics_tensor(ol, DEV)
        st["tf"], st["ws"] = B.alloc(n, Z, Y, X, mask, DEV)
        st["tiles"] = torch.empty((n, P, Z, Y, X), device=DEV)
        st["out"] = torch.empty((P, Z, case["tiles_y"] * case["core"], case["tiles_x"] * case["core"]), device=DEV)
        return st
    if op == "shared":
        st["tf"], ws1 = B.alloc(1, Z, Y, X, mask, DEV)
        B.wo_build_tf(ol[:1], 1, Z, Y, X, mask, st["tf"], ws1)
        st["ws"] = torch.zeros(B.wo_workspace_bytes(n, Z, Y, X, mask), dtype=torch.uint8, device=DEV)
    else:
        st["tf"], st["ws"] = B.alloc(n, Z, Y, X, mask, DEV)
        if op == "tf":
            st["optics"] = ol
            return st
        B.wo_build_tf(ol, n, Z, Y, X, mask, st["tf"], st["ws"])
    if op == "recon" and case["mode"] == "2d" and kinds == ("phase",):
        st["data"] = _thin_stacks(ol, Z, Y, X, gen)[:, None]
    else:
        st["data"] = _stacks(case, ol, gen)
    if op == "model":
        st["f"] = _specimen(n, kinds, Z, Y, X, ol[0], gen)
        st["d"] = torch.empty_like(st["data"])
        st["back"] = torch.empty_like(st["f"])
    else:
        st["out"] = torch.empty((n, P, Z, Y, X) if case.get("mode") != "2d" else (n, P, Y, X), device=DEV)
    return st


def run(st):
    case = st["case"]
    op = case["op"]
    if op == "train":
        B.wo_est_backward(st["wbf"], st["w"], st["feat"], st["target"], case["n"], E.SCALE, E.OFFSET, st["grad"],
                          st["loss"], st["ws"])
        return {"grad": st["grad"], "loss": st["loss"]}
    if op == "tune":
        pb = st["problem"]
        pb.evaluate()
        return {"value": pb.value, "grad": pb.grad}
    n, Z, Y, X = _shape(case)
    mode = B.WO_MODE_2D if case.get("mode") == "2d" else B.WO_MODE_3D
    if op == "predict":
        B.wo_spectrum(st["data"], None, B.WO_MODE_2D, st["spec"], n, Z, Y, X)
        B.wo_est_features(st["spec"], st["optics"], n, Z, Y, X, st["feat"])
        return {"features": st["feat"], "optics": st["est"].predict(st["feat"])}
    if op == "fused":
        B.wo_reconstruct_fused(st["tf"], case["channels"], st["data"], None, ETA, B.WO_ETA_RELATIVE, mode, st["out"],
                               n, Z, Y, X, st["ws"])
        return st["out"]
    k = st["kinds"]
    if op == "tf":
        B.wo_build_tf(st["optics"], n, Z, Y, X, k, st["tf"], st["ws"])
        spec, stats = B.tf_views(st["tf"], n, Z, Y, X, k)
        cols = [c for c, on in ((slice(0, 2), k & 3), (slice(2, 4), k & 4)) if on]
        return {"tf": spec, "maxima": [stats[:, c] for c in cols]}
    if op == "field":
        g = (Z, case["tiles_y"], case["tiles_x"], case["core"], case["halo"])
        B.wo_build_tf_device(st["optics"], n, Z, Y, X, k, st["tf"], st["ws"])
        B.wo_reconstruct_field_tiles(st["tf"], k, st["field"], *g, None, st["eta"], B.WO_ETA_RELATIVE, mode,
                                     st["tiles"], st["ws"])
        P = st["out"].shape[0]
        for p in range(P):  # one property's tiles at a time
            B.wo_tile_blend(st["tiles"] if P == 1 else st["tiles"][:, p].contiguous(), *g, st["out"][p])
        return st["out"]
    if op == "shared":
        B.wo_reconstruct_shared_tf(st["tf"], k, st["data"], None, st["eta"], B.WO_ETA_RELATIVE, mode, st["out"], n,
                                   Z, Y, X, st["ws"])
        return st["out"]
    if op == "model":
        bg = [1.0] * st["d"].shape[1]
        B.wo_forward(st["tf"], k, st["f"], bg, st["d"], n, Z, Y, X, st["ws"])
        B.wo_forward_adjoint(st["tf"], k, st["data"], bg, st["back"], n, Z, Y, X, st["ws"])
        return {"data": st["d"], "adjoint": st["back"]}
    B.wo_reconstruct(st["tf"], k, st["data"], None, st["eta"], B.WO_ETA_RELATIVE, mode, st["out"], n, Z, Y, X,
                     st["ws"])
    return st["out"]


# ------------------------------------------------------------------------ work
def _fft_flops(points, length, real=True):
    return (2.5 if real else 5.0) * points * math.log2(max(length, 2))


def work(case):
    op = case["op"]
    if op == "train":
        macs = sum((64 // r) ** 2 * co * ci * 9 for (ci, co, _), r in zip(LAYERS, (1, 2, 4, 8)))
        return {"bytes": case["n"] * (3 * 4096 * 4 + 16) + 186020 * 6 + 4, "flops": 6 * macs * case["n"]}
    n, Z, Y, X = _shape(case)
    vox, perp = n * Z * Y * X, Y * X
    half = n * Z * Y * (X // 2 + 1)
    if op == "tune":
        p = 4 if case["params"] == "all" else 1
        return {"bytes": 8 * half + n * (72 + 8 * (1 + p)),
                "flops": 2 * _fft_flops(vox, perp, False) + 2 * _fft_flops(vox, perp) + 40 * vox}
    if op == "predict":
        macs = sum((64 // r) ** 2 * co * ci * 9 for (ci, co, _), r in zip(LAYERS, (1, 2, 4, 8)))
        return {"bytes": 4 * vox + n * (3 * 4096 * 4 + 72 + 16) + 186020 * 2,
                "flops": _fft_flops(vox, perp) + 10 * half + 2 * macs * n}
    if op == "fused":
        C = case["channels"]
        out = vox if case["mode"] == "3d" else n * Y * X
        return {"bytes": C * (4 * vox + 8 * half) + 4 * out,
                "flops": (C + 1) * _fft_flops(vox, Z * perp) + 12 * C * half}
    kinds = _kinds(case)
    modes, P = _modes(kinds)
    arms = 2 * ("phase" in kinds or "absorption" in kinds) + ("fluor" in kinds)
    build = arms * _fft_flops(vox, perp, False) + P * _fft_flops(vox, Z * perp)
    if op == "tf":
        return {"bytes": 8 * P * half + n * 72, "flops": build}
    C = len(modes)
    solve = (C + P) * _fft_flops(vox, Z * perp) + 20 * P * half
    if op == "field":
        field = Z * case["tiles_y"] * case["tiles_x"] * case["core"] ** 2
        return {"bytes": 4 * field * (1 + P) + n * 72, "flops": build + solve + 10 * P * vox}
    bank = 8 * P * half // (n if op == "shared" else 1)
    if op == "model":
        return {"bytes": 2 * (4 * (C + P) * vox + bank), "flops": 2 * solve}
    out = vox if case.get("mode") != "2d" else n * Y * X
    return {"bytes": 4 * C * vox + bank + 4 * P * out, "flops": solve}


# ----------------------------------------------------------------------- exact
def _tikhonov(H, D, kinds, axes_sum=None):
    """Spectra of the properties: D[mode] the channels' spectra, regularised relative to the largest sum |H|^2."""
    modes, P = _modes(kinds)
    F = [None] * P
    for (_, ps), d in zip(modes, D):
        h2 = sum(H[k].abs() ** 2 for _, k in ps)
        if axes_sum is None:
            den = h2 + ETA * h2.max()
            for i, k in ps:
                F[i] = H[k].conj() * d / den
            continue
        # the thin object: every plane one channel, a 1 x 1 or 2 x 2 system per transverse frequency
        s = h2.sum(dim=axes_sum)
        ea = ETA * s.max()
        r = [(H[k].conj() * d).sum(dim=axes_sum) for _, k in ps]
        if len(ps) == 1:
            F[ps[0][0]] = r[0] / (s + ea)
            continue
        (i0, k0), (i1, k1) = ps
        m00 = (H[k0].abs() ** 2).sum(dim=axes_sum) + ea
        m11 = (H[k1].abs() ** 2).sum(dim=axes_sum) + ea
        m01 = (H[k0].conj() * H[k1]).sum(dim=axes_sum)
        det = m00 * m11 - m01.abs() ** 2
        F[i0] = (m11 * r[0] - m01 * r[1]) / det
        F[i1] = (m00 * r[1] - m01.conj() * r[0]) / det
    return F


def _recon64(case, optics, data):
    """Reconstructions of data [n, C, Z, Y, X] in float64."""
    n, C, Z, Y, X = data.shape
    kinds = _kinds(case)
    _, P = _modes(kinds)
    two = case.get("mode") == "2d"
    out = torch.empty((n, P, Y, X) if two else (n, P, Z, Y, X), dtype=torch.float64, device=DEV)
    for o, i, j in _each(optics):
        H = (_plane_tfs if two else _tfs)(o, Z, Y, X, kinds)
        for lo, hi in _chunks(i, j, max(1, 16000000 // (Z * Y * X))):
            d = data[lo:hi].to(torch.float64)
            d = d - d.mean(dim=(-3, -2, -1), keepdim=True)
            if two:
                F = _tikhonov(H, [torch.fft.rfft2(d[:, c]) for c in range(C)], kinds, axes_sum=-3)
                for p in range(P):
                    out[lo:hi, p] = torch.fft.irfft2(F[p], s=(Y, X))
            else:
                F = _tikhonov(H, [torch.fft.rfftn(d[:, c], dim=(-3, -2, -1)) for c in range(C)], kinds)
                for p in range(P):
                    out[lo:hi, p] = torch.fft.irfftn(F[p], s=(Z, Y, X), dim=(-3, -2, -1))
    return out


def _tune64(case, start, data):
    """Loss and gradient of every tile from the definition, the gradient by torch's reverse mode."""
    n, Z, Y, X = data.shape
    p = 4 if case["params"] == "all" else 1
    val = torch.empty(n, dtype=torch.float64, device=DEV)
    grad = torch.empty((n, p), dtype=torch.float64, device=DEV)
    w = torch.full((X // 2 + 1,), 2.0, dtype=torch.float64, device=DEV)
    w[0] = w[-1] = 1.0
    for t, o in enumerate(start):
        d = data[t].to(torch.float64)
        D = torch.fft.rfft2(d - d.mean())
        th = torch.tensor([o["defocus_um"], o["tilt_x"], o["tilt_y"], o["na_ill"]], dtype=torch.float64, device=DEV,
                          requires_grad=True)
        H = _plane_tfs(o, Z, Y, X, ("phase",), theta=tuple(th), smooth=case["params"] == "all")["phase"]
        F = (H.conj() * D).sum(dim=0) / (H.abs().square().sum(dim=0) + ETA)
        R = D - H * F
        q = (R.real ** 2 + R.imag ** 2).sum(dim=0) + ETA * (F.real ** 2 + F.imag ** 2)
        L = (w * q).sum() / (Y * X)
        (g,) = torch.autograd.grad(L, th)
        val[t], grad[t] = L.detach(), g[:p]
    return {"value": val, "grad": grad}


def _features64(optics, data):
    n, Z, Y, X = data.shape
    out = torch.zeros((n, 3, 64, 64), dtype=torch.float64, device=DEV)
    order = (torch.arange(Z, device=DEV) - Z // 2) % Z
    for t, o in enumerate(optics):
        d = data[t].to(torch.float64)
        D = torch.fft.fft2(d - d.mean())[order].reshape(Z, -1)
        ny, nx = _axis(Y, o["pixel_um"])[:, None], _axis(X, o["pixel_um"])[None, :]
        r = torch.sqrt(nx * nx + ny * ny)
        b = torch.floor(r / (2.0 * o["na_det"] / o["lambda_um"]) * 64).to(torch.int64).flatten()
        ok = b < 64
        safe = torch.where(r > 0, r, torch.ones_like(r))
        ux, uy = (nx / safe).flatten()[ok], (ny / safe).flatten()[ok]
        b, D = b[ok], D[:, ok]

        def binned(v):
            return torch.zeros((v.shape[0], 64), dtype=torch.float64, device=DEV).index_add_(1, b, v)

        P = binned(D.abs() ** 2)
        C = D[1:] * D[:-1].conj()
        den = binned(D[1:].abs() * D[:-1].abs())
        den = torch.where(den > 0, den, torch.full_like(den, math.inf))
        out[t, 0, :Z] = torch.log1p(P / P.mean())
        out[t, 1, :Z - 1] = binned(C.imag * ux) / den
        out[t, 2, :Z - 1] = binned(C.imag * uy) / den
    return out


def exact(case, seed):
    op, gen = case["op"], _gen(seed)
    scale = torch.tensor(E_SCALE, dtype=torch.float64, device=DEV)
    offset = torch.tensor(E_OFFSET, dtype=torch.float64, device=DEV)
    if op == "train":
        feat = _features(case["n"], gen)
        out, params = _network64(_weights(seed), feat, grad=True)
        tgt = (_targets(case["n"], seed + 1).to(torch.float64) - offset) / scale
        loss = ((out - tgt) ** 2).mean()
        g = torch.autograd.grad(loss, params)
        return {"grad": torch.cat([v.flatten() for v in g]), "loss": loss.detach().reshape(1)}
    if op == "fused":
        n, C, Z, Y, X = case["n"], case["channels"], case["Z"], case["Y"], case["X"]
        ol = _apertures(case, seed)
        two = case["mode"] == "2d"
        f = _specimen(n, ("phase",), Z, Y, X, OPTICS, gen)
        d = torch.empty((n, C, Z, Y, X), device=DEV)
        for t in range(n):
            for c in range(C):
                d[t, c] = _image(_tfs(ol[t * C + c], Z, Y, X, ("phase",), torch.float32), f[t:t + 1],
                                 ("phase",))[0, 0]
        d = _add_noise(d, gen)
        out = torch.empty((n, Y, X) if two else (n, Z, Y, X), dtype=torch.float64, device=DEV)
        for t in range(n):
            num = den = 0.0
            for c in range(C):
                x = d[t, c].to(torch.float64)
                x = x - x.mean()
                if two:
                    H, D = _plane_tfs(ol[t * C + c], Z, Y, X, ("phase",))["phase"], torch.fft.rfft2(x)
                    num, den = num + (H.conj() * D).sum(dim=0), den + (H.abs() ** 2).sum(dim=0)
                else:
                    H, D = _tfs(ol[t * C + c], Z, Y, X, ("phase",))["phase"], torch.fft.rfftn(x)
                    num, den = num + H.conj() * D, den + H.abs() ** 2
            F = num / (den + ETA * den.max())
            out[t] = torch.fft.irfft2(F, s=(Y, X)) if two else torch.fft.irfftn(F, s=(Z, Y, X))
        return out
    n, Z, Y, X = _shape(case)
    ol = _optics(case, seed, n)
    if op == "tune":
        return _tune64(case, _start_optics(case, ol),
                       _thin_stacks(ol, Z, Y, X, gen, smooth=case["params"] == "all"))
    if op == "predict":
        f = _features64(ol, _thin_stacks(ol, Z, Y, X, gen, smooth=True))
        return {"features": f, "optics": _network64(_weights(seed), f)[0] * scale + offset}
    kinds = _kinds(case)
    modes, P = _modes(kinds)
    if op == "tf":
        tf = torch.empty((n, P, Z, Y, X // 2 + 1), dtype=torch.complex128, device=DEV)
        maxima = [torch.empty((n, 2), dtype=torch.float64, device=DEV) for _ in modes]
        for o, i, j in _each(ol):
            H = _tfs(o, Z, Y, X, kinds)
            for m, (_, ps) in enumerate(modes):
                h2 = sum(H[k].abs() ** 2 for _, k in ps)
                maxima[m][i:j, 0], maxima[m][i:j, 1] = h2.max(), h2.sum(dim=0).max()
                for p, k in ps:
                    tf[i:j, p] = H[k]
        return {"tf": tf, "maxima": maxima}
    if op == "field":
        core, halo, e = case["core"], case["halo"], Y
        field = _field(case, ol, gen)
        Yf, Xf = field.shape[-2:]
        u = torch.arange(e, device=DEV, dtype=torch.float64) + 0.5
        w1 = torch.minimum(torch.minimum(torch.ones_like(u), u / (2 * halo)), (e - u) / (2 * halo))
        w2 = w1[:, None] * w1[None, :]
        acc = torch.zeros((P, Z, Yf, Xf), dtype=torch.float64, device=DEV)
        wsum = torch.zeros((Yf, Xf), dtype=torch.float64, device=DEV)
        for t, o in enumerate(ol):
            y0, x0 = t // case["tiles_x"] * core - halo, t % case["tiles_x"] * core - halo
            d = field[:, _window(y0, e, Yf, True)][..., _window(x0, e, Xf, True)]
            r = _recon64(case, [o], d[None, None])[0]
            ya, yb, xa, xb = max(y0, 0), min(y0 + e, Yf), max(x0, 0), min(x0 + e, Xf)
            w = w2[ya - y0:yb - y0, xa - x0:xb - x0]
            acc[..., ya:yb, xa:xb] += w * r[..., ya - y0:yb - y0, xa - x0:xb - x0]
            wsum[ya:yb, xa:xb] += w
        return acc / wsum
    if op == "recon" and case["mode"] == "2d" and kinds == ("phase",):
        return _recon64(case, ol, _thin_stacks(ol, Z, Y, X, gen)[:, None])
    data = _stacks(case, ol, gen)
    if op != "model":
        return _recon64(case, ol, data)
    f = _specimen(n, kinds, Z, Y, X, ol[0], gen)
    d = torch.empty(data.shape, dtype=torch.float64, device=DEV)
    back = torch.empty(f.shape, dtype=torch.float64, device=DEV)
    for o, i, j in _each(ol):
        H = _tfs(o, Z, Y, X, kinds)
        d[i:j] = _image(H, f[i:j].to(torch.float64), kinds)
        for c, ps in modes:
            D = torch.fft.rfftn(data[i:j, c].to(torch.float64) - 1.0, dim=(-3, -2, -1))
            for p, k in ps:
                back[i:j, p] = torch.fft.irfftn(H[k].conj() * D, s=(Z, Y, X), dim=(-3, -2, -1))
    return {"data": d, "adjoint": back}


E_SCALE, E_OFFSET = (1.0, 0.1, 0.1, 0.125), (0.0, 0.0, 0.0, 0.825)  # the estimator's output standardisation
