"""What the schedule table says is what runs: rows of 768 samples on the engine
that is pinned."""
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
