"""Inlier thresholds whose square does not fit FP32, infinity among them: the
scoring pass's upper bounds still hold, next to trials that only FP64 decides
(NaN Dopplers among their seeds).  Every output equals the oracle's."""
import numpy as np
import pytest

from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau", [np.inf, 3e19, 1e3])
@pytest.mark.parametrize("dim,H", [(2, 48), (3, 48), (2, 1024), (3, 1024)])
def test_wide_threshold(dim, H, tau):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2012_12618_gb300 import rvh
    rng = np.random.default_rng(dim * 10 + H)
    # shared-memory rows below 1536 / 2048 points, split rows above; staged from 128 / 256
    sizes = [5, 100, 300, 1500, 2050, 3000, 300, 2600]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    n = int(off[-1])
    az = rng.uniform(-1.0, 1.0, n).astype(np.float32)
    el = rng.uniform(-0.25, 0.25, n).astype(np.float32) if dim == 3 else None
    dop = rng.uniform(-30.0, 30.0, n)
    dop[rng.random(n) < 0.5] = np.nan      # most trials hold one, the first of a cluster among them
    dop[off[6]:] = rng.uniform(-1.0, 1.0, n - off[6]) * 1e10  # residuals far beyond the smallest tau
    dop = dop.astype(np.float32)
    with rvh.Context(0) as ctx:
        g = G.run_rvh(ctx, az, dop, off, el=el, H=H, tau=tau, seed=3)
    o = G.run_oracle_parallel(az, dop, off, el=el, H=H, tau=tau, seed=3)
    for k in ("inlier_count", "best_hypothesis", "status", "inlier_mask"):
        assert np.array_equal(g[k], o[k]), k
    # velocities of up to 1e10 m/s and more
    assert np.allclose(g["vx"], o["vx"], rtol=1e-6, atol=1e-6, equal_nan=True)
