"""Banks at critical sampling: NA_det / lambda one rounding below 1 / (2 pixel)
is accepted, and the rounding of k / (X pixel) then leaves the column X/2
(whose own mirror image it is) inside the detection pupil.  The passes that
store half of the columns must store that one too.

The reference is the general passes (an all-zero aberration): the even passes
differ from them by float32 rounding alone (2e-6 bounds it, see
test_gpu_even.py), the derivative banks not at all.
"""
import pytest

import phantom as ph

pytestmark = pytest.mark.gpu

# lambda, NA_det, pixel = lambda / (2 NA_det) with column X/2 inside the pupil for X = 48, 96 and 192
LAM, NA = 0.698, 0.55


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2412_09775_gb300.build import build
    build()
    from paper_2412_09775_gb300 import binding
    return binding, torch, torch.device("cuda:0")


def critical(X, **kw):
    pixel = LAM / (2 * NA)
    assert NA / LAM < 1.0 / (2.0 * pixel)  # accepted ...
    assert ((X // 2) / (X * pixel)) ** 2 <= (NA / LAM) ** 2  # ... and the column X/2 is in the pupil
    return ph.optics(lambda_um=LAM, na_det=NA, na_ill=0.0, pixel_um=pixel, z_step_um=0.5, n_medium=1.0, **kw)


def banks(env, X, Y, kinds):
    B, torch, dev = env
    ol = [critical(X, defocus_um=0.2), critical(X, defocus_um=-0.4)]
    out = []
    for general in (False, True):
        tf = torch.full((B.wo_tf_bytes(2, 3, Y, X, kinds),), 0x7F, dtype=torch.uint8, device=dev)
        ws = torch.full((B.wo_aberrated_workspace_bytes(2, 3, Y, X, kinds),), 0x7F, dtype=torch.uint8, device=dev)
        if general:
            B.wo_build_tf_aberrated(ol, [[0.0]] * 2, 2, 3, Y, X, kinds, tf, ws)
        else:
            B.wo_build_tf(ol, 2, 3, Y, X, kinds, tf, ws)
        out.append(B.tf_views(tf, 2, 3, Y, X, kinds)[0])
    return out


@pytest.mark.parametrize("X,Y", [(48, 64), (96, 96), (192, 32)])
@pytest.mark.parametrize("kinds", [4, 1, 7, 1 | 32])
def test_even_passes_store_the_nyquist_column(env, X, Y, kinds):
    _, torch, _ = env
    got, want = banks(env, X, Y, kinds)
    d = torch.linalg.vector_norm((got - want).to(torch.complex128))
    assert float(d) <= 2e-6 * float(torch.linalg.vector_norm(want.to(torch.complex128)))


@pytest.mark.parametrize("X,Y", [(48, 64), (96, 24), (192, 32)])
@pytest.mark.parametrize("kinds", [8 | 16, 64 | 32 | 16])
def test_derivative_banks_store_the_nyquist_column(env, X, Y, kinds):
    _, torch, _ = env
    got, want = banks(env, X, Y, kinds)
    assert torch.equal(got, want)
