"""Batches of many small graphs: more graphs than CTAs, more than one chunk of the
task prefix (512), team and single-CTA tasks side by side, one and two CTAs per SM in
the lazy rounds, recorded and replayed."""
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


def kinds():
    return [graphgen.barabasi_albert(300, 2, 3), graphgen.grid_road(7, 9, 0.15, 0.01, 5), graphgen.rmat(8, 3.0, seed=4),
            sg.path(40), sg.star(65), sg.complete(9), graphgen.barabasi_albert(700, 3, 1)]


@pytest.mark.parametrize("count", [1, 151, 153, 305, 511, 512, 513, 700])
def test_many(gcm, count):
    some = kinds()
    graphs = [some[i % len(some)] for i in range(count)]
    ks = [1 + (5 * i) % 8 for i in range(count)]
    want = [oracle.greedy_plain(rp, ci, 8) for rp, ci in some]
    with gcm.Batch(graphs) as B:
        for kw in ({}, {"capture": True}, {"capture": True}):
            groups, far, _ = B.greedy(ks, **kw)
            for i, (q, k) in enumerate(zip(groups, ks)):
                grp, ft, _ = want[i % len(some)]
                np.testing.assert_array_equal(q, grp[:k], err_msg=str(i))
                assert far[i] == ft[k - 1]


@pytest.mark.parametrize("many", [3, 200])
def test_with_larger_graphs(gcm, many):
    """On both sides of the sizes from which tasks go to teams (65,536 adjacency
    entries) and round 0 takes the far counts (4,096 vertices)."""
    some = kinds()
    big = [graphgen.barabasi_albert(4095, 8, 1), graphgen.barabasi_albert(4096, 8, 2), graphgen.rmat(13, 8.0, seed=3)]
    assert big[0][1].size < 1 << 16 < big[2][1].size
    for last in range(1, 4):
        graphs = [some[i % len(some)] for i in range(many)] + big[:last]
        ks = [6] * len(graphs)
        with gcm.Batch(graphs) as B:
            groups, far, _ = B.greedy(ks)
        for i, g in enumerate(graphs):
            if many <= i or i < len(some):
                with gcm.Graph(*g) as G:
                    grp, f, _ = G.greedy(6)
            else:
                grp, f = groups[i % len(some)], far[i % len(some)]
            np.testing.assert_array_equal(groups[i], grp, err_msg=str(i))
            assert far[i] == f
