"""The column, row and z passes at the lengths and edges where their kernels
differ, against the same step in float64 torch.

Bounds: a float32 transform of a few thousand points is a few 1e-7 off its
exact value (relative 2-norm); an operator is two three-dimensional ones and
a product, about 1e-6; both are allowed five times that.
"""
import numpy as np
import pytest

import phantom as ph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2412_09775_gb300.build import build
    build()
    from paper_2412_09775_gb300 import binding
    return binding, torch, torch.device("cuda:0")


def rel(torch, got, want):
    dt = torch.complex128 if want.is_complex() else torch.float64
    return float(torch.linalg.vector_norm(got.to(dt) - want) / torch.linalg.vector_norm(want))


def noise(torch, dev, seed, *shape):
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    return torch.randn(shape, generator=g, device=dev)


@pytest.mark.parametrize("Y", [2, 3, 6, 8, 12, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 2048])
@pytest.mark.parametrize("X", [2, 96, 768])
def test_plane_spectra_at_every_column_length(env, Y, X):
    """Columns of one to four stages, strips of one, 16 and a last odd column;
    rows of 768 samples."""
    B, torch, dev = env
    d = noise(torch, dev, Y, 2, 3, Y, X)
    spec = torch.empty((2, 3, Y, X // 2 + 1), dtype=torch.complex64, device=dev)
    B.wo_spectrum(d, [0.0], B.WO_MODE_2D, spec, 2, 3, Y, X)
    assert rel(torch, spec, torch.fft.rfft2(d.double())) < 1.5e-6


@pytest.mark.parametrize("kinds,Y,X", [("dz", 32, 48), ("dz", 256, 64), ("dz", 24, 128), ("dz", 64, 96),
                                       ("grad", 32, 48), ("grad", 192, 96), ("grad", 384, 64), ("grad", 48, 192)])
def test_derivative_banks_share_the_even_columns(env, kinds, Y, X):
    """B and B' stored for k_x >= 0 alone against the passes that store every
    column (an all-zero aberration): the same bits."""
    B, torch, dev = env
    k = (B.WO_TF_PHASE_DZ if kinds == "dz" else B.WO_TF_PHASE_GRAD) | B.WO_TF_PLANES
    ol = [ph.optics(na_ill=0.7, tilt_x=0.08, tilt_y=-0.05, defocus_um=0.3), ph.optics(na_ill=0.9, defocus_um=-0.2),
          ph.optics(na_ill=0.4, tilt_x=-0.6, tilt_y=0.3)]
    banks = []
    for general in (False, True):
        tf = torch.full((B.wo_tf_bytes(3, 3, Y, X, k),), 0x7F, dtype=torch.uint8, device=dev)
        ws = torch.full((B.wo_aberrated_workspace_bytes(3, 3, Y, X, k),), 0x7F, dtype=torch.uint8, device=dev)
        if general:
            B.wo_build_tf_aberrated(ol, [[0.0]] * 3, 3, 3, Y, X, k, tf, ws)
        else:
            B.wo_build_tf(ol, 3, 3, Y, X, k, tf, ws)
        banks.append(B.tf_views(tf, 3, 3, Y, X, k)[0])
    assert torch.equal(banks[0], banks[1])


def operator64(B, torch, tf, n, Z, Y, X, kinds):
    """The bank's transfer functions in 64 bits, zero outside the support, and its modes (channel, slots)."""
    H, stats = B.tf_views(tf, n, Z, Y, X, kinds)
    H = H.to(torch.complex128)
    fy = torch.fft.fftfreq(Y, dtype=torch.float64, device=H.device)[:, None]
    fx = torch.arange(X // 2 + 1, dtype=torch.float64, device=H.device)[None] / X
    r = stats[:, 5].double()[:, None, None]
    inside = (fy ** 2 + fx ** 2)[None] <= r ** 2
    H = H * inside[:, None, None]
    lf = bin(kinds & 3).count("1")
    modes = ([list(range(lf))] if lf else []) + ([[lf]] if kinds & 4 else [])
    return H, modes


# tiles of different supports: the widest past Nyquist/2, the narrowest a few columns
SETS = [dict(na_ill=0.9, defocus_um=0.2), dict(na_ill=0.1, na_det=0.3, tilt_x=0.02), dict(na_ill=0.0, na_det=0.1),
        dict(na_ill=0.5, na_det=0.9, tilt_y=0.2, defocus_um=-0.3)]


@pytest.mark.parametrize("kinds", [1, 4, 3, 5, 7])
@pytest.mark.parametrize("shape", [(12, 48, 64), (16, 64, 96), (24, 32, 768), (6, 24, 48), (8, 384, 32),
                                   (3, 512, 24), (1, 32, 48), (2, 24, 32), (4, 32, 32), (32, 6, 32), (48, 12, 32),
                                   (64, 8, 32), (96, 6, 48), (128, 6, 32), (192, 4, 32), (256, 4, 32)])
def test_operators_by_shape_and_kinds(env, kinds, shape):
    """Forward, adjoint and reconstructions (3D and 2D) of tiles with different
    supports, with a workspace of NaNs: no pass may read what no pass wrote.
    Register and shared-memory rows, z columns of one to three stages, strips
    that cross rows or end partly filled."""
    B, torch, dev = env
    Z, Y, X = shape
    n = len(SETS)
    ol = [ph.optics(**s) for s in SETS]
    tf, _ = B.alloc(n, Z, Y, X, kinds, dev)
    ws = torch.full((B.wo_workspace_bytes(n, Z, Y, X, kinds),), 0xFF, dtype=torch.uint8, device=dev)
    ws[:256].zero_()
    B.wo_build_tf(ol, n, Z, Y, X, kinds, tf, ws)
    H, modes = operator64(B, torch, tf, n, Z, Y, X, kinds)
    P, C = H.shape[1], len(modes)
    f, d = noise(torch, dev, 1, n, P, Z, Y, X), noise(torch, dev, 2, n, C, Z, Y, X)
    F, D = torch.fft.rfftn(f.double(), dim=(-3, -2, -1)), torch.fft.rfftn(d.double(), dim=(-3, -2, -1))
    inv = lambda s: torch.fft.irfftn(s, s=(Z, Y, X), dim=(-3, -2, -1))

    ws[256:].fill_(0xFF)
    got = torch.empty_like(d)
    B.wo_forward(tf, kinds, f, None, got, n, Z, Y, X, ws)
    want = torch.stack([inv(sum(H[:, p] * F[:, p] for p in m)) for m in modes], dim=1)
    assert rel(torch, got, want) < 5e-6
    ws[256:].fill_(0xFF)
    got = torch.empty_like(f)
    B.wo_forward_adjoint(tf, kinds, d, None, got, n, Z, Y, X, ws)
    want = torch.empty_like(f, dtype=torch.float64)
    for c, m in enumerate(modes):
        for p in m:
            want[:, p] = inv(H[:, p].conj() * D[:, c])
    assert rel(torch, got, want) < 5e-6
    eta = 0.5  # absolute; the spectra are white, so a small one would only measure the bank's own zeros
    ws[256:].fill_(0xFF)
    B.wo_reconstruct(tf, kinds, d, [0.0] * C, [eta] * C, B.WO_ETA_ABSOLUTE, B.WO_MODE_3D, got, n, Z, Y, X, ws)
    for c, m in enumerate(modes):
        den = sum(H[:, p].abs() ** 2 for p in m) + eta
        for p in m:
            want[:, p] = inv(H[:, p].conj() * D[:, c] / den)
    assert rel(torch, got, want) < 5e-6
    if kinds in (1, 4, 5):  # one property a mode: the 2D solve is a quotient of sums over k_z
        ws[256:].fill_(0xFF)
        got2 = torch.empty((n, P, Y, X), device=dev)
        B.wo_reconstruct(tf, kinds, d, [0.0] * C, [eta] * C, B.WO_ETA_ABSOLUTE, B.WO_MODE_2D, got2, n, Z, Y, X, ws)
        want2 = torch.stack([torch.fft.irfft2((H[:, m[0]].conj() * D[:, c]).sum(1)
                                              / ((H[:, m[0]].abs() ** 2).sum(1) + Z * eta), s=(Y, X))
                             for c, m in enumerate(modes)], dim=1)
        assert rel(torch, got2, want2) < 5e-6


@pytest.mark.parametrize("Z,E", [(16, 64), (48, 128)])
def test_plane_engine_by_support(env, Z, E):
    """The same for kx-major banks, one a tile and one for all."""
    B, torch, dev = env
    n, k = len(SETS), 1 | B.WO_TF_KX_MAJOR
    ol = [ph.optics(**s) for s in SETS]
    d = noise(torch, dev, 3, n, 1, Z, E, E)
    D = torch.fft.rfftn(d.double(), dim=(-3, -2, -1))
    for shared in (False, True):
        m = 1 if shared else n
        tf, _ = B.alloc(m, Z, E, E, k, dev)
        ws = torch.full((B.wo_workspace_bytes(n, Z, E, E, k),), 0xFF, dtype=torch.uint8, device=dev)
        ws[:256].zero_()
        B.wo_build_tf(ol[3:] if shared else ol, m, Z, E, E, k, tf, ws)
        H, _ = operator64(B, torch, tf, m, Z, E, E, k)
        ws[256:].fill_(0xFF)
        got = torch.empty_like(d)
        call = B.wo_reconstruct_shared_tf if shared else B.wo_reconstruct
        call(tf, k, d, [0.0], [0.5], B.WO_ETA_ABSOLUTE, B.WO_MODE_3D, got, n, Z, E, E, ws)
        assert B.wo_sync_status(ws)[0] == 0
        want = torch.fft.irfftn(H.conj() * D / (H.abs() ** 2 + 0.5), s=(Z, E, E), dim=(-3, -2, -1))
        assert rel(torch, got, want) < 5e-6


@pytest.mark.parametrize("mode", ["3d", "2d"])
@pytest.mark.parametrize("Z", [8, 12, 16, 24, 32, 48, 64, 96, 128])
def test_fusion_at_every_plane_count(env, Z, mode):
    """Register columns (12 to 64, 128) and shared-memory ones, a last partial CTA, relative regulariser."""
    B, torch, dev = env
    n, C, Y, X = 2, 3, 6, 32
    ol = [ph.optics(na_ill=0.15, tilt_x=0.5 * np.cos(a), tilt_y=0.5 * np.sin(a)) for a in range(n * C)]
    tf, ws0 = B.alloc(n * C, Z, Y, X, "phase", dev)
    B.wo_build_tf(ol, n * C, Z, Y, X, "phase", tf, ws0)
    H = B.tf_views(tf, n * C, Z, Y, X, 1)[0].to(torch.complex128).reshape(n, C, Z, Y, X // 2 + 1)
    d = noise(torch, dev, Z, n, C, Z, Y, X)
    D = torch.fft.rfftn(d.double(), dim=(-3, -2, -1))
    D[..., 0, 0, 0] = 0  # the default background is the channel's mean
    ws = torch.full((B.wo_fused_workspace_bytes(C, n, Z, Y, X),), 0xFF, dtype=torch.uint8, device=dev)
    two = mode == "2d"
    out = torch.empty((n, Y, X) if two else (n, Z, Y, X), device=dev)
    B.wo_reconstruct_fused(tf, C, d, None, 0.05, B.WO_ETA_RELATIVE, B.WO_MODE_2D if two else B.WO_MODE_3D, out, n, Z,
                           Y, X, ws)
    num, den = (H.conj() * D).sum(1), (H.abs() ** 2).sum(1)
    if two:
        num, den = num.sum(1), den.sum(1)
    lam = 0.05 * den.amax(dim=tuple(range(1, den.dim())), keepdim=True)
    want = torch.fft.irfftn(num / (den + lam), s=(Y, X) if two else (Z, Y, X), dim=(-2, -1) if two else (-3, -2, -1))
    assert rel(torch, out, want) < 5e-6
