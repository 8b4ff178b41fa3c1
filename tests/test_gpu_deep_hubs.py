"""Deep graphs with long rows: the bounds that pass from hop to hop go through rows
of a thread, of a warp and of a CTA.  Groups and top-k sets against the 64-lane
batches."""
import numpy as np
import pytest

from paper_1710_01144_gb300 import graphgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gcm():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1710_01144_gb300 import build, gc

    build.build()
    return gc


def csr(n, u, v):
    key = np.unique(np.concatenate([u, v]).astype(np.int64) * n + np.concatenate([v, u]))
    src, dst = key // n, key % n
    keep = src != dst
    rp = np.concatenate([[0], np.cumsum(np.bincount(src[keep], minlength=n))])
    return rp.astype(np.int32), dst[keep].astype(np.int32)


def edges(g):
    u = np.repeat(np.arange(g[0].size - 1), np.diff(g[0]))
    return u[u < g[1]], g[1][u < g[1]]


def with_leaves(g, at, leaves):
    """`leaves` new vertices at each vertex of `at`."""
    u, v = edges(g)
    n = g[0].size - 1
    at = np.repeat(at, leaves)
    return csr(n + at.size, np.concatenate([u, at]), np.concatenate([v, n + np.arange(at.size)]))


@pytest.mark.parametrize("side,at,leaves", [(90, [4000], 32), (90, [4000, 17], 33), (90, [9], 2047), (90, [9], 2600),
                                            (100, [5000, 5001, 30], 4100)])
def test_bounds_through_long_rows(gcm, side, at, leaves):
    g = with_leaves(graphgen.grid_road(side, side, 0.2, 0.01, 3), at, leaves)
    with gcm.Graph(*g) as G:
        want, f, _ = G.greedy(8, round0_lanes=-1)
        got, f2, _ = G.greedy(8)
        np.testing.assert_array_equal(got, want)
        assert f == f2
        ids, far, _ = G.top_closeness(25)
        ids0, far0, _ = G.top_closeness(25, round0_lanes=-1)
        np.testing.assert_array_equal(ids, ids0)
        np.testing.assert_array_equal(far, far0)
