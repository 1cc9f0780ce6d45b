"""The estimator's features by the number of rows at work (tiles times planes):
one row a block while they all fit the chip, four from there on, and blocks
past the stack.  Against the float64 reference at the bounds of the other
features tests, and the times of short and few stacks beside larger ones."""
import numpy as np
import pytest

import phantom as ph
from oracle import estimator as OE

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2412_09775_gb300.build import build
    build()
    from paper_2412_09775_gb300 import binding
    return binding, torch, torch.device("cuda:0")


# 760 rows are the last that take one block each
@pytest.mark.parametrize("n,shape", [(190, (4, 48, 64)), (191, (4, 48, 64)), (384, (2, 48, 64)), (130, (6, 48, 96)),
                                     (12, (64, 64, 32)), (256, (3, 128, 48))])
def test_features_by_rows(env, n, shape):
    B, torch, dev = env
    Z, Y, X = shape
    two = [dict(o, smooth_source=True) for o in ph.tile_optics(np.random.default_rng(4), 2)]
    d = np.stack([1 + 0.01 * ph.uniform_volume(10 + t, shape) for t in range(2)]).astype(np.float32)
    data = torch.tensor(d, device=dev)[torch.arange(n, device=dev) % 2].contiguous()
    spec = torch.empty((n, Z, Y, X // 2 + 1), dtype=torch.complex64, device=dev)
    B.wo_spectrum(data, None, B.WO_MODE_2D, spec, n, Z, Y, X)
    feat = torch.full((n, 3, 64, 64), np.nan, dtype=torch.float32, device=dev)
    B.wo_est_features(spec, B.optics_tensor([two[t % 2] for t in range(n)], dev), n, Z, Y, X, feat)
    got = feat.cpu().numpy()
    for t in range(2):
        want = OE.tile_features(d[t].astype(np.float64), two[t])
        assert np.abs(got[t::2, 0] - want[0]).max() <= 1e-4 * max(1.0, np.abs(want[0]).max())
        assert np.abs(got[t::2, 1:] - want[1:]).max() <= 1e-3


def time_of(env, n, Z, Y, X):
    B, torch, dev = env
    spec = torch.randn((n, Z, Y, X // 2 + 1), dtype=torch.complex64, device=dev)
    o, feat = B.optics_tensor([ph.optics()] * n, dev), torch.empty((n, 3, 64, 64), device=dev)
    best = 1e9
    B.wo_profile_enable(True)
    for _ in range(6):
        B.wo_profile_read()
        for _ in range(5):
            B.wo_est_features(spec, o, n, Z, Y, X, feat)
        torch.cuda.synchronize()
        best = min(best, B.wo_profile_read()["est_features"][1])
    B.wo_profile_enable(False)
    return best


def test_rows_past_the_stack_cost_nothing(env):
    """60 of 64 rows past a stack of 4 planes: a sixteenth of the work of 64 planes."""
    assert time_of(env, 1024, 4, 32, 32) <= 0.25 * time_of(env, 1024, 64, 32, 32)


def test_one_tile_does_not_wait_for_one_warp_a_row(env):
    """One tile leaves most of the chip idle: its time is a row's walk, which a
    block shares among its warps (0.21 of 64 tiles' time; 0.39 by one warp)."""
    assert time_of(env, 1, 48, 128, 128) <= 0.3 * time_of(env, 64, 48, 128, 128)
