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


def with_tail(g, length, at):
    """A path of `length` new vertices at vertex `at`."""
    u, v = edges(g)
    n = g[0].size - 1
    t = n + np.arange(length)
    return csr(n + length, np.concatenate([u, [at], t[:-1]]), np.concatenate([v, t]))


def broom(length, leaves):
    return with_leaves(with_tail((np.zeros(2, np.int32), np.zeros(0, np.int32)), length - 1, 0), [length - 1], leaves)


@pytest.mark.parametrize("name,g,far", [
    ("attachment with a tail", with_tail(graphgen.barabasi_albert(6000, 3, 3), 40, 5999), False),
    ("tree with a tail", with_tail(graphgen.barabasi_albert(30000, 1, 3), 40, 29999), False),
    ("rmat with a tail", with_tail(graphgen.rmat(14, 3.0, seed=4), 45, 5), False),
    ("broom", broom(70, 6000), False),
    ("road", graphgen.grid_road(50, 50, 0.2, 0.01, 3), True),
    ("road with leaves", with_leaves(graphgen.grid_road(60, 60, 0.2, 0.01, 3), [9, 700], 500), True)])
def test_a_tail_does_not_make_a_graph_deep(gcm, name, g, far):
    """All have more than 32 BFS levels; only where distances are long too do the
    one-source searches take over (and then evaluate other candidates)."""
    import oracle

    k = 5
    grp, ft, _, _ = oracle.greedypp(*g, k)
    with gcm.Graph(*g) as G:
        got, f, st = G.greedy(k)
        ref, _, st0 = G.greedy(k, round0_lanes=-1)
        ids, far_, _ = G.top_closeness(12)
        ids0, far0, _ = G.top_closeness(12, round0_lanes=-1)
    np.testing.assert_array_equal(got, grp)
    np.testing.assert_array_equal(ref, grp)
    assert f == ft[-1]
    np.testing.assert_array_equal(ids, ids0)
    np.testing.assert_array_equal(far_, far0)
    assert (st["evals"] != st0["evals"]) == far
