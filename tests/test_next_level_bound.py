"""The BFScut bound with a cap on the next level (farness mode of csrc/gc_cta.cuh
and csrc/gc_grid.cuh), restated in numpy and checked against the oracle's
distances: after level d, at most D = sum over the vertices at distance d of
(deg - 1) vertices are at distance d + 1, so
    f({v}) >= s + (d + 1) min(rest, D) + (d + 2) (rest - min(rest, D))
with s the distances counted and rest the vertices not reached.  And the whole
round 0 on graphs whose every vertex survives the degree bound."""
import numpy as np
import pytest

import oracle
from paper_1710_01144_gb300 import graphgen
from tests import smallgraphs as sg


def cases():
    return [("path40", sg.path(40)), ("cycle31", sg.cycle(31)), ("star30", sg.star(30)), ("k9", sg.complete(9)),
            ("tree", sg.tree_random(400, 3)), ("gnp", sg.gnp_connected(150, 0.03, 5)),
            ("ba1", graphgen.barabasi_albert(500, 1, 2)), ("ba2", graphgen.barabasi_albert(600, 2, 7)),
            ("rmat10", graphgen.rmat(10, 3.0, seed=3)), ("road", graphgen.grid_road(30, 27, 0.2, 0.01, 5))]


@pytest.mark.parametrize("name,g", cases())
def test_bound_is_a_lower_bound(name, g):
    rp, ci = g
    n, deg = rp.size - 1, np.diff(rp).astype(np.int64)
    for v in np.random.default_rng(3).choice(n, size=min(n, 40), replace=False):
        dist = oracle.bfs(rp, ci, [int(v)]).astype(np.int64)
        f = int(dist.sum())
        for d in range(1, int(dist.max()) + 1):
            s, rest = int(dist[dist <= d].sum()), int((dist > d).sum())
            nx = min(rest, int((deg[dist == d] - 1).sum()))
            assert int((dist == d + 1).sum()) <= nx
            assert s + (d + 1) * nx + (d + 2) * (rest - nx) <= f


@pytest.mark.gpu
@pytest.mark.parametrize("n,m,k", [(65, 1, 3), (700, 2, 5), (6000, 2, 8), (5000, 3, 300)])
def test_round0_on_flat_graphs(n, m, k):
    """gc_greedy (64-lane CTA and grid batches) and top-k closeness."""
    import torch

    from paper_1710_01144_gb300 import build, gc

    assert torch.cuda.is_available()
    build.build()
    rp, ci = graphgen.barabasi_albert(n, m, 11)
    ids, far, _ = oracle.topk_closeness(rp, ci, min(k, 60))
    grp, ft, _, _ = oracle.greedypp(rp, ci, 3)
    with gc.Graph(rp, ci) as G:
        for lanes in (0, -1):
            got, f, _ = G.greedy(3, round0_lanes=lanes)
            np.testing.assert_array_equal(got, grp)
            assert f == ft[-1]
            ti, tf, _ = G.top_closeness(min(k, 60), round0_lanes=lanes)
            np.testing.assert_array_equal(ti, ids)
            np.testing.assert_array_equal(tf, far)
