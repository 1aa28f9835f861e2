"""The heading's arctangent against the host's in long double (GPU; builds
tests/cuda/heading_exact.cu): within 3 x 2^-52 of the angle, as stated.  Its
own bound: the table entries' and the product's roundings move the tangent by
at most (sqrt(2) + 1) 2^-54, the last sum rounds by at most 2^-52 (angles from
2 on), and the terms of the tangent, below 2^-7.9, by less than 2^-59: 1.7."""
import os
import subprocess

import pytest

from paper_2012_12618_gb300 import build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_heading_within_its_bound(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    exe = str(tmp_path / "heading_exact")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, os.path.join(HERE, "cuda", "heading_exact.cu"), "-o", exe],
                   check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    d = dict(kv.split("=") for kv in r.stdout.split())
    print(r.stdout)
    assert int(d["points"]) == 1 << 20 and int(d["worst"]) <= 3000, d
