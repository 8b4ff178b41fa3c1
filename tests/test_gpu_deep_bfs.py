"""BFS of graphs so deep that one CTA takes level after level: distances across
several of its stretches of 256 levels, and waits that stay short of the time
limit however deep the graph is."""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("n", [2, 255, 256, 257, 258, 511, 513, 5000])
def test_farness_of_paths(gcm, n):
    rp, ci = sg.path(n)
    with gcm.Graph(rp, ci) as G:
        for s in (0, n // 2, n - 1):
            assert G.farness([s]) == s * (s + 1) // 2 + (n - 1 - s) * (n - s) // 2


@pytest.mark.parametrize("name,g", [("grid3x700", sg.grid(3, 700)), ("caterpillar", sg.caterpillar(900, 2)),
                                    ("fan", sg.caterpillar(300, 20))])
def test_farness_and_updates(gcm, name, g):
    rp, ci = g
    n = rp.size - 1
    grp, ft, _ = oracle.greedy_plain(rp, ci, 3)
    with gcm.Graph(rp, ci) as G:
        for S in ([0], [n - 1], [0, n // 3, n - 1]):
            assert G.farness(S) == oracle.farness(rp, ci, S)
        got, f, _ = G.greedy(3)  # d_S lowered over most of the graph
        np.testing.assert_array_equal(got, grp)
        assert f == ft[-1]


def test_no_wait_grows_with_the_depth(gcm):
    """8,192 levels of 2 us each against a limit of 4 ms a wait."""
    rp, ci = sg.path(8192)
    with gcm.Graph(rp, ci) as G:
        want, f, _ = G.greedy(2)
        got, f2, _ = G.greedy(2, timeout_us=4000)
    np.testing.assert_array_equal(got, want)
    assert f == f2 and got[0] == 4095
