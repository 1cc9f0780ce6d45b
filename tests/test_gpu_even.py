"""The TF passes for an even detection pupil (tilted, on-axis and smooth
sources) against the general passes.

A build with an all-zero aberration takes the general passes on the same
optics; the two banks differ by float32 rounding alone: both round the same
transforms, about 1e-7 of the largest value each (the general passes' own
distance to the float64 oracle is a few 1e-7), so 2e-6 relative bounds them.
"""
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


def optics_set(n):
    """Tilted and on-axis tiles in turn, sources from a point to the whole detection pupil."""
    sets = [dict(na_ill=0.7, tilt_x=0.08, tilt_y=-0.05, defocus_um=0.3), dict(na_ill=0.9, defocus_um=-0.2),
            dict(na_ill=0.0, tilt_x=-0.4, defocus_um=0.1), dict(na_ill=1.2, tilt_y=0.05),
            dict(na_ill=0.4, tilt_x=-0.6, tilt_y=0.3, defocus_um=-0.6)]
    return [ph.optics(**sets[i % len(sets)]) for i in range(n)]


def both(env, ol, shape, kinds):
    B, torch, dev = env
    Z, Y, X = shape
    n = len(ol)
    out = []
    for general in (False, True):
        tf = torch.full((B.wo_tf_bytes(n, Z, Y, X, kinds),), 0x7F, dtype=torch.uint8, device=dev)
        ws = torch.full((B.wo_aberrated_workspace_bytes(n, Z, Y, X, kinds),), 0x7F, dtype=torch.uint8, device=dev)
        if general:
            B.wo_build_tf_aberrated(ol, [[0.0]] * n, n, Z, Y, X, kinds, tf, ws)
        else:
            B.wo_build_tf(ol, n, Z, Y, X, kinds, tf, ws)
        torch.cuda.synchronize()
        out.append(B.tf_views(tf, n, Z, Y, X, kinds)[0])
    return out


def check(env, ol, shape, kinds):
    _, torch, _ = env
    got, want = both(env, ol, shape, kinds)
    for t in range(len(ol)):
        for k in range(got.shape[1]):
            d = torch.linalg.vector_norm((got[t, k] - want[t, k]).to(torch.complex128))
            assert float(d) <= 2e-6 * float(torch.linalg.vector_norm(want[t, k].to(torch.complex128))), (t, k)


@pytest.mark.parametrize("kinds", [1, 2, 4, 3, 5, 7, 1 | 32])
@pytest.mark.parametrize("shape", [(3, 32, 48), (2, 64, 192), (1, 192, 32)])
def test_even_passes_match_the_general_ones(env, kinds, shape):
    """Every kind set, tiles mixed within warps and an odd number of them."""
    check(env, optics_set(5), shape, kinds)


@pytest.mark.parametrize("Y,X", [(48, 64), (96, 96), (128, 256), (256, 128), (512, 64), (64, 512), (192, 192)])
def test_even_passes_at_every_row_and_column_length(env, Y, X):
    check(env, optics_set(3), (2, Y, X), 7)


@pytest.mark.parametrize("kind", [1, 4])
@pytest.mark.parametrize("Z,E", [(48, 192), (32, 128), (16, 64)])
def test_even_passes_write_kx_major_banks(env, kind, Z, E):
    B, torch, dev = env
    ol = optics_set(3)
    std, _ = both(env, ol, (Z, E, E), kind)
    tf, ws = B.alloc(3, Z, E, E, kind | B.WO_TF_KX_MAJOR, dev)
    B.wo_build_tf(ol, 3, Z, E, E, kind | B.WO_TF_KX_MAJOR, tf, ws)
    assert B.wo_sync_status(ws)[0] == 0
    got = B.tf_views(tf, 3, Z, E, E, kind | B.WO_TF_KX_MAJOR)[0]
    for t in range(3):
        d = torch.linalg.vector_norm((got[t] - std[t]).to(torch.complex128))
        assert float(d) <= 2e-6 * float(torch.linalg.vector_norm(std[t].to(torch.complex128))), t
