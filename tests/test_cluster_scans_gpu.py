"""The clustering stage's device-wide scans at the edges of their ranges:
one tile of the scan holds 2048 values, and the CSR offsets of up to 4096
clusters come from one block, of more from the tiled scan.  The points are
well-separated groups on a line whose sizes are known, in shuffled order, so
the labels (groups numbered by their smallest core index), the permutation
and the offsets are known without an oracle and must be identical."""
import numpy as np
import pytest

from paper_2012_12618_gb300 import rvh
from tests import test_cluster_gpu as C

pytestmark = pytest.mark.gpu
torch, ctx = C.torch, C.ctx  # the module's fixtures


@pytest.mark.parametrize("n_groups,extra,min_pts", [
    (1, 0, 1), (1, 0, 2), (2047, 0, 1), (2048, 0, 1), (2049, 0, 1),
    (4095, 2, 1), (4096, 2, 1), (4097, 2, 1), (8192, 1, 1), (8193, 1, 1), (6145, 3, 2)])
def test_group_counts(torch, ctx, n_groups, extra, min_pts):
    rng = np.random.default_rng(n_groups + extra)
    size = 1 + np.arange(n_groups) % (extra + 1)
    group = rng.permutation(np.repeat(np.arange(n_groups), size))
    feats = (10.0 * group + 0.25 * rng.random(group.size)).astype(np.float32)
    kept = size[group] >= min_pts          # a group's points are all neighbours of one another
    want = np.full(group.size, -1)
    first, inv = np.unique(group[kept], return_index=True)[1], np.unique(group[kept], return_inverse=True)[1]
    want[kept] = np.argsort(np.argsort(first))[inv]
    nc = first.size
    rc, got_nc, lab, perm, off = C._cluster(torch, ctx, feats, 1.0, min_pts)
    assert rc == rvh.RVH_OK and got_nc == nc
    assert np.array_equal(lab, want)
    p, offs = C._csr(want, nc)
    assert np.array_equal(off[:nc + 1], offs)
    assert np.array_equal(perm[:p.size], p)
