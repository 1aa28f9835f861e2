"""The 3D refinement's residuals in pairs of FP32 stay within their bound of
the FP64 ones (GPU; builds tests/cuda/low_residual.cu)."""
import os
import subprocess

import pytest

from paper_2012_12618_gb300 import build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_residual_bound(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    exe = str(tmp_path / "low_residual")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, os.path.join(HERE, "cuda", "low_residual.cu"), "-o", exe],
                   check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    d = dict(kv.split("=") for kv in r.stdout.split())
    assert int(d["points"]) == 1 << 22 and int(d["bad"]) == 0, d
    assert 0.3 < float(d["worst"]) <= 1.0, d  # the bound is met, and not by orders of magnitude
