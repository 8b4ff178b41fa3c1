"""bitGreedy++ on both sides of the size up to which a CTA holds its targets'
words in shared memory, at the edges of a 32-target word, and with rows longer
than a warp."""
import numpy as np
import pytest

import oracle
from paper_1710_01144_gb300 import graphgen
from tests import smallgraphs as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,g,k", [("n1", (np.zeros(2, np.int32), np.zeros(0, np.int32)), 1),
                                      ("path2", sg.path(2), 2), ("path31", sg.path(31), 5), ("path33", sg.path(33), 33),
                                      ("star1500", sg.star(1500), 4), ("path1100", sg.path(1100), 3),
                                      ("ba15999", graphgen.barabasi_albert(15999, 2, 3), 4),
                                      ("ba16000", graphgen.barabasi_albert(16000, 2, 3), 4),
                                      ("ba16001", graphgen.barabasi_albert(16001, 2, 3), 4)])
def test_bits_sizes(name, g, k):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1710_01144_gb300 import build, gc

    build.build()
    rp, ci = g
    with gc.Graph(rp, ci) as G:
        got, f, _ = G.greedy_bits(k)
        again, f2, _ = G.greedy_bits(k)
        if name.startswith("ba"):
            want, ft, _ = G.greedy(k)
        else:
            want, ft, _ = oracle.greedy_plain(rp, ci, k)
            ft = int(ft[-1])
    np.testing.assert_array_equal(got, want)
    np.testing.assert_array_equal(again, want)
    assert f == f2 == ft


def test_bits_disconnected():
    from paper_1710_01144_gb300 import gc

    rp, ci = sg.disjoint_union(sg.path(40), sg.path(3))
    with gc.Graph(rp, ci) as G:
        with pytest.raises(gc.GcError) as e:
            G.greedy_bits(2)
        assert e.value.code == gc.GC_EDISCONNECTED
