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


@pytest.mark.parametrize("n,E,limit", [(61, 128, 1.95), (15, 256, 1.63)])
def test_one_volume_of_24_planes(env, n, E, limit):
    """1.66 and 1.38 row passes in shared memory, 2.24 and 1.89 through registers:
    the limits lie halfway."""
    B, torch, dev = env
    _, tf, ws = bank(env, 1, n, 24, E)
    d, out = torch.randn((n, 1, 24, E, E), device=dev), torch.empty((n, 1, 24, E, E), device=dev)
    t = times(env, lambda: B.wo_reconstruct(tf, 1, d, None, [1e-3], B.WO_ETA_RELATIVE, B.WO_MODE_3D, out, n, 24, E, E, ws))
    assert t["z_fused"] <= limit * t["rows_r2c"], t


@pytest.mark.parametrize("kinds,n,Z,E", [(7, 1, 96, 512), (3, 12, 24, 256), (5, 19, 16, 256)])
def test_tf_z_pass_leaves_the_empty_columns_out(env, kinds, n, Z, E):
    """A grid eight times as fine: the transfer functions fill an eighth of the
    columns, and the z pass takes a small part of its time on the full grid."""
    t = []
    for px in (0.1, 0.0125):
        B = env[0]
        ol, tf, ws = bank(env, kinds, n, Z, E, pixel_um=px)
        t.append(times(env, lambda: B.wo_build_tf(ol, n, Z, E, E, kinds, tf, ws))["tf_zpass"])
    assert t[1] <= 0.4 * t[0], t


def test_tf_z_pass_of_128_planes(env):
    """Two kinds: 1.6 times the y pass's time in shared memory, 2.1 times through registers."""
    B = env[0]
    ol, tf, ws = bank(env, 3, 9, 128, 128)
    t = times(env, lambda: B.wo_build_tf(ol, 9, 128, 128, 128, 3, tf, ws))
    assert t["tf_zpass"] <= 1.85 * t["tf_ypass"], t


@pytest.mark.parametrize("kinds", [3, 5, 7, 8])
@pytest.mark.parametrize("Z", [2, 6, 12, 16, 24, 48, 64, 128, 192])
@pytest.mark.parametrize("px", [0.1, 0.02])
def test_tf_z_pass_at_both_walks(env, kinds, Z, px):
    """Rows cut at the support (optics on the host) and whole rows (optics on the
    device, extent unknown): the same bits in the columns of both, and each
    bank's statistics those of its values."""
    B, torch, dev = env
    n, Y, X = 2, 24, 96
    ol = [ph.optics(na_ill=0.6, tilt_x=0.1, pixel_um=px, z_step_um=0.05), ph.optics(na_ill=0.2, na_det=0.5, pixel_um=px, z_step_um=0.05)]
    host, ws = B.alloc(n, Z, Y, X, kinds, dev)
    devb = torch.empty_like(host)
    ws[256:].fill_(0xFF)
    B.wo_build_tf(ol, n, Z, Y, X, kinds, host, ws)          # rows cut at x_cols
    B.wo_build_tf_device(B.optics_tensor(ol, dev), n, Z, Y, X, kinds, devb, ws)  # optics unknown: whole rows
    H, st = B.tf_views(host, n, Z, Y, X, kinds)
    D, sd = B.tf_views(devb, n, Z, Y, X, kinds)
    cols = int(max((1.2 + min(1.2, 0.7)) / 0.532 * X * px, (1.2 if kinds & 4 else 0) * 2 / 0.532 * X * px)) + 2
    assert torch.equal(H[..., :cols], D[..., :cols])
    lf = 1 if kinds == 8 else bin(kinds & 3).count("1")
    p = (D.to(torch.complex128).abs() ** 2)
    for s, slots in ((0, range(lf)), (2, [lf] if kinds & 4 else [])):
        if not list(slots):
            continue
        q = sum(p[:, k] for k in slots)  # [n, Z, Y, Xh]
        for stats in (st, sd):
            assert torch.allclose(stats[:, s].double(), q.amax((1, 2, 3)), rtol=1e-5)
            assert torch.allclose(stats[:, s + 1].double(), q.sum(1).amax((1, 2)), rtol=1e-5)
