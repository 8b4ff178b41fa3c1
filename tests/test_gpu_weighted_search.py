"""The weighted searches in distance order (csrc/gc_weighted.cu): bucketed round
0 with its cut, rows ordered by weight (one to three counting passes), distances
in shared memory at 512 and 1024 threads and in global memory, handles of
different sizes in one process.  Groups against the oracle where it is quick;
unit weights against gc_greedy on the larger graphs."""
import numpy as np
import pytest

import oracle
from paper_1710_01144_gb300 import graphgen
from tests import smallgraphs as sg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gcm():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1710_01144_gb300 import build, gc

    build.build()
    return gc


@pytest.mark.parametrize("w_max", [1, 3, 255, 256, 70000])
@pytest.mark.parametrize("name,g", [("ba1025", graphgen.barabasi_albert(1025, 3, 2)), ("star1200", sg.star(1200)),
                                    ("rmat11", graphgen.rmat(11, 6.0, seed=4)),
                                    ("road36", graphgen.grid_road(36, 36, 0.2, 0.01, 3)), ("path5", sg.path(5))])
def test_groups_match_oracle(gcm, name, g, w_max):
    rp, ci = g
    w = graphgen.edge_weights(rp, ci, w_max, 7)
    k = min(6, rp.size - 1)
    grp, ft, _ = oracle.wgreedy_plain(rp, ci, w, k)
    with gcm.Graph(rp, ci) as G:
        G.set_weights(w, validate=True)
        for _ in range(2):  # the workspaces are at rest again
            got, f, st = G.greedy_weighted(k)
            np.testing.assert_array_equal(got, grp)
            assert f == ft[-1] and st["round0_evals"] == rp.size - 1


@pytest.mark.parametrize("n", [24001, 47999, 48001])
def test_large_graphs_with_unit_weights(gcm, n):
    rp, ci = graphgen.barabasi_albert(n, 8 if n == 24001 else 2, 5)
    small = graphgen.barabasi_albert(1500, 3, 1)
    with gcm.Graph(rp, ci) as G, gcm.Graph(*small) as H:
        G.set_weights(np.full(ci.size, 3, np.int32))
        H.set_weights(np.ones(small[1].size, np.int32))
        first = G.greedy_weighted(3)
        h = H.greedy_weighted(4)  # another size in between
        again = G.greedy_weighted(3)
        ref = G.greedy(3)
        np.testing.assert_array_equal(h[0], H.greedy(4)[0])
    for got in (first, again):
        np.testing.assert_array_equal(got[0], ref[0])
        assert got[1] == 3 * ref[1]
