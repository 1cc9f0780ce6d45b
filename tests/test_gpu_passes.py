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
