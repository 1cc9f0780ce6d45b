"""The fusion kernels in the WO_CHECK variant of the library (as
test_gpu_check_build.py does for the other families): clean statuses and the
normal library's bits, with register and shared-memory z columns, both modes
and a last partial block."""
import os
import subprocess
import sys

import numpy as np
import pytest

import phantom as ph

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys, numpy as np, torch
sys.path.insert(0, {root!r}); sys.path.insert(0, {tests!r})
from paper_2412_09775_gb300.build import build
build(check=True)
from paper_2412_09775_gb300 import binding as B
assert B.wo_check_build()
import test_gpu_check_fusion as T
np.savez({path!r}, **T.run(B, torch, torch.device("cuda:0")))
"""


def run(B, torch, dev):
    out = {}
    n, C, Y, X = 2, 3, 6, 32
    ol = [ph.optics(na_ill=0.15, tilt_x=0.5 * np.cos(a), tilt_y=0.5 * np.sin(a)) for a in range(n * C)]
    for Z in (8, 16):
        tf, ws0 = B.alloc(n * C, Z, Y, X, "phase", dev)
        B.wo_build_tf(ol, n * C, Z, Y, X, "phase", tf, ws0)
        d = torch.from_numpy(ph.uniform_volume(3, (n, C, Z, Y, X), 0.9, 1.1).astype(np.float32)).to(dev)
        ws = torch.zeros(B.wo_fused_workspace_bytes(C, n, Z, Y, X), dtype=torch.uint8, device=dev)
        for mode, shape in ((B.WO_MODE_3D, (n, Z, Y, X)), (B.WO_MODE_2D, (n, Y, X))):
            f = torch.empty(shape, device=dev)
            B.wo_reconstruct_fused(tf, C, d, None, 0.05, B.WO_ETA_RELATIVE, mode, f, n, Z, Y, X, ws)
            assert B.wo_sync_status(ws) == (0, 0, 0)
            out[f"{Z} {mode}"] = f.cpu().numpy()
    return out


def test_fusion_in_the_check_build(tmp_path):
    import torch
    from paper_2412_09775_gb300.build import build
    build()
    from paper_2412_09775_gb300 import binding as B
    path = str(tmp_path / "fused.npz")
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, tests=os.path.join(ROOT, "tests"), path=path)],
                       env=dict(os.environ, WO_LIB="check"), capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stderr[-3000:]
    got, want = np.load(path), run(B, torch, torch.device("cuda:0"))
    assert not B.wo_check_build()
    for k, v in want.items():
        assert np.array_equal(got[k], v), k
