"""The estimator's features at the edges of their kernel (a number of
planes that ends inside a group of four rows, all 64 rows, ragged point
counts), against the float64 reference at the bounds of the other features test."""
import numpy as np
import pytest

import phantom as ph
from oracle import estimator as OE

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(2, 48, 64), (6, 48, 96), (64, 64, 32), (3, 128, 48)])
def test_features_at_ragged_shapes(shape):
    import torch
    from paper_2412_09775_gb300.build import build
    build()
    from paper_2412_09775_gb300 import binding as B
    dev = torch.device("cuda:0")
    Z, Y, X = shape
    ol = [dict(o, smooth_source=True) for o in ph.tile_optics(np.random.default_rng(4), 2)]
    d = np.stack([1 + 0.01 * ph.uniform_volume(10 + t, shape) for t in range(2)]).astype(np.float32)
    spec = torch.empty((2, Z, Y, X // 2 + 1), dtype=torch.complex64, device=dev)
    B.wo_spectrum(torch.tensor(d, device=dev), None, B.WO_MODE_2D, spec, 2, Z, Y, X)
    feat = torch.full((2, 3, 64, 64), np.nan, dtype=torch.float32, device=dev)
    B.wo_est_features(spec, B.optics_tensor(ol, dev), 2, Z, Y, X, feat)
    got = feat.cpu().numpy()
    for t in range(2):
        want = OE.tile_features(d[t].astype(np.float64), ol[t])
        assert np.abs(got[t, 0] - want[0]).max() <= 1e-4 * max(1.0, np.abs(want[0]).max())
        assert np.abs(got[t, 1:] - want[1:]).max() <= 1e-3
