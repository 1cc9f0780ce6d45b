"""The z passes that come in two forms (through registers or in shared memory):
at the lengths where the rule changes form, the times of the form that runs
beside a row pass of the same call.  Values: test_gpu_passes.py and the parity
tests, at every length."""
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


def times(env, call):
    B, torch, _ = env
    best = {}
    B.wo_profile_enable(True)
    for _ in range(6):
        B.wo_profile_read()
        for _ in range(5):
            call()
        torch.cuda.synchronize()
        for k, v in B.wo_profile_read().items():
            best[k] = min(best.get(k, 1e9), v[1])
    B.wo_profile_enable(False)
    return best


def bank(env, kinds, n, Z, E, **kw):
    B, torch, dev = env
    ol = [ph.optics(na_ill=0.8, tilt_x=0.05 * (t % 3), defocus_um=0.1 * (t % 5), **kw) for t in range(n)]
    tf, ws = B.alloc(n, Z, E, E, kinds, dev)
    B.wo_build_tf(ol, n, Z, E, E, kinds, tf, ws)
    return ol, tf, ws


@pytest.mark.parametrize("n,E", [(61, 128), (15, 256)])
def test_one_volume_of_24_planes(env, n, E):
    """1.35 to 1.6 row passes in shared memory, 1.9 to 2.1 through registers."""
    B, torch, dev = env
    _, tf, ws = bank(env, 1, n, 24, E)
    d, out = torch.randn((n, 1, 24, E, E), device=dev), torch.empty((n, 1, 24, E, E), device=dev)
    t = times(env, lambda: B.wo_reconstruct(tf, 1, d, None, [1e-3], B.WO_ETA_RELATIVE, B.WO_MODE_3D, out, n, 24, E, E, ws))
    assert t["z_fused"] <= 1.75 * t["rows_r2c"], t
