"""What the schedule table and its built-in rules say is what runs: rows of 768
samples on the engine that is pinned, few planes of 64 x 64 on the fused x-y
kernels, also after the autotuner has seen a large batch."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2412_09775_gb300.build import build
    build()
    from paper_2412_09775_gb300 import binding
    return binding, torch, torch.device("cuda:0")


def profile(env, call, reps=5):
    """Best total milliseconds of each kernel family over a few rounds of the call."""
    B, torch, _ = env
    best = {}
    B.wo_profile_enable(True)
    for _ in range(6):
        B.wo_profile_read()
        for _ in range(reps):
            call()
        torch.cuda.synchronize()
        for k, v in B.wo_profile_read().items():
            best[k] = min(best.get(k, 1e9), v[1])
    B.wo_profile_enable(False)
    return best


def test_rows_of_768_run_on_the_pinned_engine(env):
    """The shared-memory rows take 1.7 times the register rows; both give the
    float64 spectra to 1.5e-6."""
    B, torch, dev = env
    n, Z, Y, X = 2, 24, 384, 768
    d = torch.randn((n, Z, Y, X), device=dev)
    want = torch.fft.rfft2(d.double())
    t = {}
    for e in (B.WO_ENGINE_SMEM, B.WO_ENGINE_HYBRID):
        B.wo_schedule_set(B.WO_PASS_ROWS, X // 2, e)
        try:
            spec = torch.empty((n, Z, Y, X // 2 + 1), dtype=torch.complex64, device=dev)
            call = lambda: B.wo_spectrum(d, [0.0], B.WO_MODE_2D, spec, n, Z, Y, X)
            t[e] = profile(env, call)["rows_r2c"]
            err = torch.linalg.vector_norm(spec.to(torch.complex128) - want) / torch.linalg.vector_norm(want)
            assert float(err) < 1.5e-6
        finally:
            B.wo_schedule_set(B.WO_PASS_ROWS, X // 2, B.WO_ENGINE_DEFAULT)
    assert t[B.WO_ENGINE_SMEM] > 1.25 * t[B.WO_ENGINE_HYBRID], t


def small_stacks(env, n, Z):
    """A reconstruction of n stacks of Z x 64 x 64 and the data it takes."""
    import phantom as ph
    B, torch, dev = env
    tf, ws = B.alloc(n, Z, 64, 64, "phase", dev)
    one, _ = B.alloc(1, Z, 64, 64, "phase", dev)
    o = ph.optics(na_ill=0.7)
    B.wo_build_tf([o], 1, Z, 64, 64, "phase", one, ws)
    d = torch.randn((n, 1, Z, 64, 64), device=dev)
    out = torch.empty_like(d)
    call = lambda: B.wo_reconstruct_shared_tf(one, "phase", d, [0.0], [0.5], B.WO_ETA_ABSOLUTE, B.WO_MODE_3D, out, n, Z,
                                              64, 64, ws)
    return call, d, out, B.tf_views(one, 1, Z, 64, 64, 1), ws


@pytest.mark.parametrize("n,Z,fused", [(1, 16, True), (48, 16, True), (49, 16, False), (256, 3, True), (384, 2, True),
                                       (385, 2, False)])
def test_few_planes_take_the_fused_xy_kernels_by_default(env, n, Z, fused):
    """On both sides of 768 planes, against float64 (the bound of the other
    operator tests)."""
    B, torch, dev = env
    call, d, out, (H, st), _ = small_stacks(env, n, Z)
    t = profile(env, call, reps=1)
    assert ("xy_fwd" in t) == fused and ("xy_inv" in t) == fused and ("rows_r2c" in t) != fused, t
    H = H.to(torch.complex128)
    f = torch.fft.fftfreq(64, dtype=torch.float64, device=dev)
    inside = f[:, None] ** 2 + (torch.arange(33, dtype=torch.float64, device=dev)[None] / 64) ** 2 <= float(st[0, 5]) ** 2
    H = H * inside
    D = torch.fft.rfftn(d.double(), dim=(-3, -2, -1))
    want = torch.fft.irfftn(H.conj() * D / (H.abs() ** 2 + 0.5), s=(Z, 64, 64), dim=(-3, -2, -1))
    assert float(torch.linalg.vector_norm(out - want) / torch.linalg.vector_norm(want)) < 5e-6


def test_tuning_a_large_batch_leaves_small_ones_their_default(env):
    """wo_autotune on many planes keeps the separate passes there; a later
    single stack must not be pinned to them."""
    B, torch, dev = env
    try:
        *_, ws = small_stacks(env, 512, 16)
        B.wo_autotune(512, 16, 64, 64, "phase", ws)
        call, *_ = small_stacks(env, 1, 16)
        assert "xy_fwd" in profile(env, call, reps=1)
    finally:
        for p, n in ((B.WO_PASS_XY, 64), (B.WO_PASS_COLS, 64), (B.WO_PASS_COLS, 16), (B.WO_PASS_ROWS, 32)):
            B.wo_schedule_set(p, n, B.WO_ENGINE_DEFAULT)
