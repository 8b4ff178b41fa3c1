"""The grid BFS and its three ways to take a level (csrc/gc_bfs.cu): bottom-up on
hub graphs, local levels on deep ones, back to a list when a small frontier is
left after bottom-up levels, and graphs that mix them.  Farness and greedy (whose
checks compare every update's decrease) against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1710_01144_gb300 import graphgen
from tests import smallgraphs as sg

pytestmark = pytest.mark.gpu


def glue(a, b):
    """Graph a with graph b hung on a's last vertex."""
    (ra, ca), (rb, cb) = a, b
    n, m = ra.size - 1, rb.size - 1
    u = np.concatenate([np.repeat(np.arange(n), np.diff(ra)), n + np.repeat(np.arange(m), np.diff(rb)), [n - 1, n]])
    v = np.concatenate([ca, cb + n, [n, n - 1]])
    o = np.lexsort((v, u))
    rp = np.concatenate([[0], np.cumsum(np.bincount(u, minlength=n + m))]).astype(np.int32)
    return rp, v[o].astype(np.int32)


def cases():
    return [("n1", (np.zeros(2, np.int32), np.zeros(0, np.int32))), ("path700", sg.path(700)), ("star5000", sg.star(5000)),
            ("k90", sg.complete(90)), ("rmat14", graphgen.rmat(14, 16.0, seed=3)),
            ("ba6000m9", graphgen.barabasi_albert(6000, 9, 4)), ("road90", graphgen.grid_road(90, 90, 0.2, 0.01, 3)),
            ("lollipop", glue(graphgen.barabasi_albert(4000, 12, 3), sg.path(400))),
            ("dumbbell", glue(glue(graphgen.barabasi_albert(3000, 12, 3), sg.path(60)),
                              graphgen.barabasi_albert(3000, 12, 8))),
            ("ends_in_star", glue(glue(graphgen.rmat(12, 16.0, seed=2), sg.path(5)), sg.star(3000)))]


@pytest.mark.parametrize("name,g", cases())
def test_farness_and_greedy(name, g):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1710_01144_gb300 import build, gc

    build.build()
    rp, ci = g
    n = rp.size - 1
    rng = np.random.default_rng(2)
    with gc.Graph(rp, ci) as G:
        for s in (1, 1, 3, min(n, 200)):
            S = rng.choice(n, min(s, n), replace=False).astype(np.int32)
            assert G.farness(S) == oracle.farness(rp, ci, S)
        assert G.farness([0]) == oracle.farness(rp, ci, [0])
        assert n < 2 or G.farness([n - 1, n - 1]) == oracle.farness(rp, ci, [n - 1])
        assert G.farness(np.argsort(-np.diff(rp), kind="stable")[:1]) == oracle.farness(
            rp, ci, np.argsort(-np.diff(rp), kind="stable")[:1].astype(np.int32))
        k = min(n, 5)
        grp, ft, _, _ = oracle.greedypp(rp, ci, k)
        got, f, _ = G.greedy(k)
        np.testing.assert_array_equal(got, grp)
        assert f == ft[-1]


def test_unreached_vertices_are_reported():
    from paper_1710_01144_gb300 import gc

    rp, ci = sg.disjoint_union(graphgen.barabasi_albert(3000, 12, 3), sg.path(7))
    with gc.Graph(rp, ci) as G:
        with pytest.raises(gc.GcError) as e:
            G.farness([5])
        assert e.value.code == gc.GC_EDISCONNECTED and "7 of 3007" in str(e.value)
        assert G.farness([5, 3001]) > 0
