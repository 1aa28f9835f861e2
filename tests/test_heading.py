"""The heading's arctangent against the library's (GPU; builds
tests/cuda/heading.cu): within 3 x 2^-52 of the angle and the library's own
error of two units in the last place of an angle up to pi."""
import os
import subprocess

import pytest

from paper_2012_12618_gb300 import build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_heading_accuracy(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    exe = str(tmp_path / "heading")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, os.path.join(HERE, "cuda", "heading.cu"), "-o", exe],
                   check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    d = dict(kv.split("=") for kv in r.stdout.split())
    print(r.stdout)
    # 3 units of 2^-52 here; the library's 2 ulp are 4 more (an ulp is 2 of them from 2 rad on)
    assert int(d["points"]) == 1 << 24 and float(d["worst"]) <= 7.0, d
    assert int(d["diff"]) == 0, d
