"""The relative regulariser of a fused reconstruction at every split of its
statistics pass (channels of one, up to four and up to sixteen; planes fewer
and more than the warps and loads of a column), against float64 torch at the
bound of the other fusion tests; and its time beside the transforms."""
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


def setup(env, n, C, Z, Y, X):
    B, torch, dev = env
    ol = [ph.optics(na_ill=0.15, tilt_x=0.5 * np.cos(a), tilt_y=0.5 * np.sin(a)) for a in range(n * C)]
    tf, ws = B.alloc(n * C, Z, Y, X, "phase", dev)
    B.wo_build_tf(ol, n * C, Z, Y, X, "phase", tf, ws)
    g = torch.Generator(device=dev)
    g.manual_seed(Z)
    d = torch.randn((n, C, Z, Y, X), generator=g, device=dev)
    return tf, d, torch.zeros(B.wo_fused_workspace_bytes(C, n, Z, Y, X), dtype=torch.uint8, device=dev)


@pytest.mark.parametrize("mode", ["3d", "2d"])
@pytest.mark.parametrize("C,Z", [(1, 2), (1, 16), (1, 48), (1, 192), (2, 3), (4, 4), (4, 24), (5, 1), (9, 6), (16, 2), (16, 32)])
def test_statistics_by_channels_and_planes(env, C, Z, mode):
    B, torch, dev = env
    n, Y, X = 2, 12, 48  # 300 columns: whole and partial groups
    tf, d, ws = setup(env, n, C, Z, Y, X)
    H = B.tf_views(tf, n * C, Z, Y, X, 1)[0].to(torch.complex128).reshape(n, C, Z, Y, X // 2 + 1)
    D = torch.fft.rfftn(d.double(), dim=(-3, -2, -1))
    D[..., 0, 0, 0] = 0
    two = mode == "2d"
    out = torch.empty((n, Y, X) if two else (n, Z, Y, X), device=dev)
    B.wo_reconstruct_fused(tf, C, d, None, 0.05, B.WO_ETA_RELATIVE, B.WO_MODE_2D if two else B.WO_MODE_3D, out, n, Z,
                           Y, X, ws)
    num, den = (H.conj() * D).sum(1), (H.abs() ** 2).sum(1)
    if two:
        num, den = num.sum(1), den.sum(1)
    lam = 0.05 * den.amax(dim=tuple(range(1, den.dim())), keepdim=True)
    want = torch.fft.irfftn(num / (den + lam), s=(Y, X) if two else (Z, Y, X), dim=(-2, -1) if two else (-3, -2, -1))
    assert float(torch.linalg.vector_norm(out - want) / torch.linalg.vector_norm(want)) < 5e-6


@pytest.mark.parametrize("n,C,Z,E", [(91, 1, 8, 128), (366, 2, 4, 64)])
def test_statistics_cost_no_more_than_a_row_pass_and_a_half(env, n, C, Z, E):
    """Read once, the bank takes the time of reading half of what a row pass
    moves; one atomic per warp and 32 columns took four to five times that."""
    B, torch, dev = env
    tf, d, ws = setup(env, n, C, Z, E, E)
    out = torch.empty((n, Z, E, E), device=dev)
    best = {}
    B.wo_profile_enable(True)
    for _ in range(6):
        B.wo_profile_read()
        for _ in range(5):
            B.wo_reconstruct_fused(tf, C, d, None, 0.05, B.WO_ETA_RELATIVE, B.WO_MODE_3D, out, n, Z, E, E, ws)
        torch.cuda.synchronize()
        for k, v in B.wo_profile_read().items():
            best[k] = min(best.get(k, 1e9), v[1])
    B.wo_profile_enable(False)
    assert best["fuse_stats"] <= 1.5 * best["rows_r2c"], best
