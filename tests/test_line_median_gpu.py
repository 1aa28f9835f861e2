"""The line model's medians and FP32 line records at their edges, against the
oracle: thresholds bit for bit, masks, counts and winners equal."""
import numpy as np
import pytest

import oracle
from paper_2012_12618_gb300 import synth
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _cluster(kind, n, rng):
    az = rng.uniform(-1.0, 1.0, n)
    dop = 10.0 * np.cos(az) - 6.0 * np.sin(az) + rng.normal(0.0, 0.05, n)
    out = rng.random(n) < 0.2
    dop = np.where(out, rng.uniform(0.0, 24.0, n), dop)
    if kind == "quantised":  # few distinct Dopplers: more keys in the middle bins than the list holds
        dop = np.round(dop / 8.0) * 8.0
    elif kind == "grid":     # a radar's Doppler bins: ties, a few keys per bin
        dop = np.round(dop / 0.1) * 0.1
    elif kind == "far":      # one far point: all others share the lowest histogram bins
        dop[0] = 3e6
    elif kind == "columns":  # few azimuths: seeds that share x or nearly do
        az = np.round(az * 2.0) / 2.0 + rng.integers(0, 2, n) * 1e-5
    elif kind == "nan":
        dop[rng.integers(0, n, max(1, n // 8))] = np.nan
    return az.astype(np.float32), dop.astype(np.float32)


@pytest.mark.parametrize("kind", ["plain", "quantised", "grid", "far", "columns", "nan"])
def test_median_and_records(kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2012_12618_gb300 import rvh
    rng = np.random.default_rng(len(kind))
    # odd and even counts, around one thread round, the list, the row capacity and the Dopplers kept in shared memory
    sizes = [2, 3, 255, 256, 257, 511, 512, 513, 1024, 1100, 2047, 2048, 2049, 2432, 2433, 4001]
    parts = [_cluster(kind, n, rng) for n in sizes]
    az, dop = (np.concatenate([p[i] for p in parts]) for i in range(2))
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    t = [torch.from_numpy(x).cuda() for x in (az, dop, off)]
    outs = rvh.alloc_outputs(len(sizes), len(az), "cuda", threshold=True)
    with rvh.Context(0) as ctx:
        ctx.check(rvh.rvh_estimate(ctx.handle, rvh.make_frame(*t),
                                   rvh.make_params(2, 1024, 0.1, 7, hypothesis_model=rvh.RVH_MODEL_PAPER_LINE),
                                   rvh.make_result(outs), None), "rvh_estimate")
        torch.cuda.synchronize()
    g = {k: v.cpu().numpy() for k, v in outs.items()}
    o = oracle.estimate(az, dop, off, num_hypotheses=1024, tau=0.1, seed=7, want_fragile=True, line_model=True)
    assert np.array_equal(g["threshold"], o["threshold"], equal_nan=True)
    rep = G.compare(g, o, off)
    assert not rep["mismatch"] and not rep["ties"], (rep["mismatch"] + rep["ties"])[:10]
