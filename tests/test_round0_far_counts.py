"""The counting bound of round 0 (k_far_counts in csrc/gc_bfs.cu): low-degree
vertices that no path of two hops can reach lift the degree bound on f({v}).
Restated here in numpy and checked against the oracle: the counted vertices
never outnumber those at distance >= 3, the bound never exceeds the exact
farness, and it is at least the degree bound."""
import numpy as np
import pytest

import oracle
from paper_1710_01144_gb300 import graphgen
from tests import smallgraphs as sg

FAR_DEG = 8


def cases():
    return [("n1", (np.zeros(2, np.int32), np.zeros(0, np.int32))), ("path2", sg.path(2)), ("path40", sg.path(40)),
            ("star30", sg.star(30)), ("k9", sg.complete(9)), ("cater", sg.caterpillar(12, 3)),
            ("tree", sg.tree_random(400, 3)), ("gnp", sg.gnp_connected(150, 0.03, 5)),
            ("ba1", graphgen.barabasi_albert(500, 1, 2)), ("ba9", graphgen.barabasi_albert(300, 9, 2)),
            ("rmat12", graphgen.rmat(12, 16.0, seed=1)), ("road", graphgen.grid_road(30, 27, 0.2, 0.01, 5))]


def far_count_bound(rp, ci):
    """(far, LB with the far counts, LB without) of every vertex."""
    n = rp.size - 1
    deg = np.diff(rp).astype(np.int64)
    src = np.repeat(np.arange(n), deg)

    def nbr_sum(x):
        out = np.zeros(n, np.int64)
        np.add.at(out, src, x[ci])
        return out

    two_hop, rest = nbr_sum(deg - 1), n - 1 - deg
    far = np.zeros(n, np.int64)
    for member in ((deg >= 1) & (deg <= 2), (deg >= 3) & (deg <= FAR_DEG)):
        cnt = nbr_sum(member.astype(np.int64))
        far += np.maximum(0, int(member.sum()) - member - cnt - nbr_sum(cnt))
    c2, c2f = np.minimum(two_hop, rest), np.minimum(two_hop, rest - np.minimum(far, rest))
    return far, deg + 2 * c2f + 3 * (rest - c2f), deg + 2 * c2 + 3 * (rest - c2)


@pytest.mark.parametrize("name,g", cases())
def test_far_counts_never_exceed_the_far_vertices(name, g):
    rp, ci = g
    n = rp.size - 1
    far, lb, lb0 = far_count_bound(rp, ci)
    assert np.all(lb >= lb0)
    for v in np.random.default_rng(5).choice(n, size=min(n, 60), replace=False):
        dist = oracle.bfs(rp, ci, [int(v)]).astype(np.int64)
        assert far[v] <= int((dist >= 3).sum())
        assert lb[v] <= int(dist.sum())


@pytest.mark.gpu
@pytest.mark.parametrize("scale,ef", [(9, 4.0), (13, 3.0), (16, 6.0), (17, 16.0)])
def test_top_closeness_with_and_without_the_counts(scale, ef):
    """The counts are part of the far-vertex probe: on and off give the same
    vertices and farness values, from one vertex to hundreds."""
    import torch

    from paper_1710_01144_gb300 import build, gc

    assert torch.cuda.is_available()
    build.build()
    rp, ci = graphgen.rmat(scale, ef, seed=4)
    with gc.Graph(rp, ci) as G:
        for k in (1, 7, 150):
            ids, far, _ = G.top_closeness(k)
            ids0, far0, _ = G.top_closeness(k, r0_probe=False)
            np.testing.assert_array_equal(ids, ids0)
            np.testing.assert_array_equal(far, far0)
        assert far0[0] == oracle.farness(rp, ci, [int(ids0[0])])
