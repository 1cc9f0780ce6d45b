"""kx-major banks with an aberrated detection pupil: the general arm and PSF-row
passes' kx-major stores, which every other kx-major bank leaves to the passes
of an even pupil.  An all-zero aberration against those (they differ by float32
rounding alone, 2e-6 as in test_gpu_even.py), and an aberration of several
terms against the float64 oracle (1e-4 as in test_gpu_aberrated.py)."""
import numpy as np
import pytest

import phantom as ph
from conftest import rel_l2
from oracle import optics as OO

pytestmark = pytest.mark.gpu

SHAPES = [(16, 64), (32, 128), (48, 192)]
TERMS = [0.0, 0.0, 0.0, 0.1, -0.15, 0.2, 0.08, -0.12, 0.0, 0.0, 0.1]


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2412_09775_gb300.build import build
    build()
    from paper_2412_09775_gb300 import binding
    return binding, torch, torch.device("cuda:0")


def optics():
    return [ph.optics(na_ill=0.8, tilt_x=0.04, tilt_y=-0.02, defocus_um=0.3), ph.optics(na_ill=0.6, defocus_um=-0.5),
            ph.optics(na_ill=0.0, tilt_x=-0.4)]  # an odd number of tiles: pairs of rows across tiles and tails


def aberrated(env, ol, zern, Z, E, kinds):
    B, torch, dev = env
    n = len(ol)
    tf = torch.full((B.wo_tf_bytes(n, Z, E, E, kinds),), 0x7F, dtype=torch.uint8, device=dev)
    ws = torch.full((B.wo_aberrated_workspace_bytes(n, Z, E, E, kinds),), 0x7F, dtype=torch.uint8, device=dev)
    ws[:256].zero_()
    B.wo_build_tf_aberrated(ol, [zern] * n, n, Z, E, E, kinds, tf, ws)
    assert B.wo_sync_status(ws)[0] == 0
    return B.tf_views(tf, n, Z, E, E, kinds)[0]


@pytest.mark.parametrize("kind", [1, 2, 4])
@pytest.mark.parametrize("Z,E", SHAPES)
def test_zero_aberration_equals_the_plain_bank(env, kind, Z, E):
    B, torch, dev = env
    k = kind | B.WO_TF_KX_MAJOR
    ol = optics()
    got = aberrated(env, ol, [0.0], Z, E, k)
    tf, ws = B.alloc(3, Z, E, E, k, dev)
    B.wo_build_tf(ol, 3, Z, E, E, k, tf, ws)
    want = B.tf_views(tf, 3, Z, E, E, k)[0]
    for t in range(3):
        d = torch.linalg.vector_norm((got[t] - want[t]).to(torch.complex128))
        assert float(d) <= 2e-6 * float(torch.linalg.vector_norm(want[t].to(torch.complex128))), t


@pytest.mark.parametrize("kind", ["phase", "absorption", "fluor"])
@pytest.mark.parametrize("Z,E", SHAPES)
def test_aberrated_kx_major_bank_matches_oracle(env, kind, Z, E):
    B = env[0]
    ol = optics()
    got = aberrated(env, ol, TERMS, Z, E, B.KIND_BITS[kind] | B.WO_TF_KX_MAJOR).cpu().numpy()
    for t in range(2):
        ref = OO.half_spectrum(OO.transfer_functions(dict(ol[t], zernike=TERMS), (Z, E, E), (kind,))[kind])
        assert rel_l2(got[t, 0], ref) <= 1e-4, t
