"""The staged scoring pass on what its histograms have to leave out (NaN and
infinite Dopplers, azimuths and elevations), and its counters."""
import numpy as np
import pytest

from paper_2012_12618_gb300 import rvh
from tests import gpu_util as G

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


def _frame(sizes, dim, rng):
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    n = int(off[-1])
    az = rng.uniform(-1.0, 1.0, n)
    el = rng.uniform(-0.25, 0.25, n) if dim == 3 else np.zeros(n)
    dop = 11.0 * np.cos(az) * np.cos(el) - 6.0 * np.sin(az) * np.cos(el) + 2.0 * np.sin(el)
    dop += rng.normal(0.0, 0.05, n)
    out = rng.random(n) < 0.2
    dop[out] = rng.uniform(-30.0, 30.0, int(out.sum()))
    return off, az.astype(np.float32), el.astype(np.float32) if dim == 3 else None, dop.astype(np.float32)


@pytest.mark.parametrize("dim,H,line", [(2, 1024, False), (3, 1024, False), (2, 1500, False), (3, 1500, False),
                                        (2, 1024, True)])
def test_values_no_trial_holds(ctx, dim, H, line):
    rng = np.random.default_rng(100 * dim + H + line)
    sizes = [127, 128, 130, 255, 256, 300, 511, 700, 1536, 2047, 2060] * 2 + [256, 260, 400, 1600]
    off, az, el, dop = _frame(sizes, dim, rng)
    for c in range(len(sizes)):
        p = np.arange(off[c], off[c + 1])
        pick = rng.permutation(p)
        k = max(1, len(p) // 50)
        dop[pick[:k]] = np.nan
        az[pick[k:2 * k]] = np.nan if c % 2 else np.inf
        if el is not None:
            el[pick[2 * k:3 * k]] = -np.inf if c % 2 else np.nan
        if c >= 22:  # an infinite Doppler makes every band infinite: FP64 decides all of the cluster
            dop[pick[3 * k]] = np.inf if c % 2 else -np.inf
        if c == 21:  # no usable direction at all
            az[p] = np.nan
    kw = dict(el=el, H=H, tau=0.1, seed=11)
    g = G.run_rvh(ctx, az, dop, off, line_model=line, **kw)
    assert rvh.rvh_set_pruning(ctx.handle, 0) == 0
    try:
        u = G.run_rvh(ctx, az, dop, off, line_model=line, **kw)
    finally:
        rvh.rvh_set_pruning(ctx.handle, 1)
    for k in G.OUT_KEYS:
        assert np.array_equal(g[k], u[k], equal_nan=g[k].dtype.kind == "f"), k
    o = G.run_oracle_parallel(az, dop, off, line_model=line, **kw)
    rep = G.compare(g, o, off)
    if line:
        assert not rep["mismatch"], rep["mismatch"][:10]
    else:
        G.check_parity(rep, tau=0.1)


@pytest.mark.parametrize("dim,H", [(2, 1024), (3, 1024), (2, 2300), (3, 2300)])
def test_staged_counters_add_up(ctx, dim, H):
    """The counts of a frame estimated in ranges of clusters add up to the
    whole frame's, and no warp's pairs are missing: every staged cluster
    scores its first stage for nearly every trial."""
    import torch
    rng = np.random.default_rng(dim + H)
    sizes = rng.integers(256, 2300, 60)
    off, az, el, dop = _frame(sizes, dim, rng)

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

    whole = counters(0, 60)
    parts = sum(counters(a, b) for a, b in ((0, 1), (1, 27), (27, 60)))
    assert np.array_equal(whole, parts), (whole, parts)
    assert whole[3] >= 60  # the lead or the winner of every cluster is counted
    first_stage = 128 if dim == 2 else 64
    # 1024 trials form a chunk; of a random pair of directions within +-1 rad fewer than one in 1000 is singular
    assert 0.95 * 60 * 1024 * first_stage < whole[4] < 0.9 * int(sizes.sum()) * H, whole
