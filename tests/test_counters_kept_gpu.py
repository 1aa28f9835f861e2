"""The launch counters outlive the scratch: after a call that the memory
budget refuses, which gives the old scratch back, the statistics are still
those of the last estimate, and the next estimates count from zero."""
import numpy as np
import pytest

from paper_2012_12618_gb300 import rvh, synth

pytestmark = pytest.mark.gpu

FIELDS = ("hypotheses", "candidates", "band_points", "fp64_hypotheses", "refined_hypotheses", "pairs_scored")


def test_statistics_after_a_refused_call():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda", 0)
    w = synth.WORKLOADS["dense3d"]

    def call(ctx, n_clusters):
        f = synth.make_frame(w, n_clusters=n_clusters, gen_seed=3)
        t = [torch.from_numpy(x).to(dev) for x in (f.azimuth, f.elevation, f.doppler, f.offsets)]
        outs = rvh.alloc_outputs(f.n_clusters, f.n_points, dev)
        rc = rvh.rvh_estimate(ctx.handle, rvh.make_frame(t[0], t[2], t[3], t[1]), rvh.make_params(3, 128, w.tau, 5),
                              rvh.make_result(outs), None)
        torch.cuda.synchronize()
        return rc

    def stats(ctx):
        s = rvh.rvh_stats()
        ctx.check(rvh.rvh_get_stats(ctx.handle, s), "stats")
        return np.array([getattr(s, k) for k in FIELDS], dtype=np.int64)

    # the rows of 16 clusters fit beside the CTAs' slots (41 MB), those of 4096 (100 MB more) do not
    with rvh.Context(0, mem_budget_bytes=96 << 20) as ctx:
        assert call(ctx, 16) == rvh.RVH_OK
        want = stats(ctx)
        assert want[4] > 0 and want[5] > 0
        assert call(ctx, 4096) == rvh.RVH_ENOMEM
        assert np.array_equal(stats(ctx), want)
        for _ in range(3):  # both copies of the counters, the first one again
            assert call(ctx, 16) == rvh.RVH_OK
            assert np.array_equal(stats(ctx), want)
