"""The kernel's counters, kept per warp: the counts of a frame estimated in
ranges of clusters add up to the whole frame's, and without pruning the
pairs scored are exactly N x H."""
import numpy as np
import pytest

from paper_2012_12618_gb300 import rvh

pytestmark = pytest.mark.gpu

FIELDS = ("fp64_hypotheses", "refined_hypotheses", "band_points", "candidates", "pairs_scored")


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = rvh.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("dim,H", [(2, 200), (3, 200), (2, 1100), (3, 1100)])
def test_counters_add_up(ctx, dim, H):
    import torch
    rng = np.random.default_rng(dim + H)
    sizes = rng.integers(1, 90, 70)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    n = int(off[-1])
    az = rng.uniform(-1.0, 1.0, n).astype(np.float32)
    az[off[40]:] = 0.3 + 1e-3 * az[off[40]:]        # far objects: 2D trials refine too
    el = rng.uniform(-0.25, 0.25, n).astype(np.float32) if dim == 3 else None
    dop = (9.0 * np.cos(az) + 4.0 * np.sin(az) + rng.normal(0.0, 0.05, n)).astype(np.float32)

    def counters(c0, c1):
        p0, p1 = off[c0], off[c1]
        e = None if el is None else el[p0:p1]
        dev = torch.device("cuda", 0)
        t = [None if x is None else torch.from_numpy(np.ascontiguousarray(x)).to(dev)
             for x in (az[p0:p1], e, dop[p0:p1], off[c0:c1 + 1] - p0)]
        outs = rvh.alloc_outputs(c1 - c0, int(p1 - p0), dev)
        ctx.check(rvh.rvh_estimate(ctx.handle, rvh.make_frame(t[0], t[2], t[3], t[1]),
                                   rvh.make_params(dim, H, 0.1, 8, first_cluster=c0), rvh.make_result(outs), None),
                  "estimate")
        torch.cuda.synchronize()
        s = rvh.rvh_stats()
        assert rvh.rvh_get_stats(ctx.handle, s) == 0
        return np.array([getattr(s, f) for f in FIELDS], dtype=np.int64)

    assert rvh.rvh_set_pruning(ctx.handle, 0) == 0
    try:
        whole = counters(0, 70)
        parts = sum(counters(a, b) for a, b in ((0, 1), (1, 33), (33, 70)))
    finally:
        rvh.rvh_set_pruning(ctx.handle, 1)
    assert np.array_equal(whole, parts), (whole, parts)
    assert whole[1] > 0
    usable = sizes[sizes >= dim]
    assert whole[4] == int(usable.sum()) * H
