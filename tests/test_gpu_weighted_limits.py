"""Weighted searches at the largest path lengths that are accepted: (n - 1) x max
weight = 2^30 - 2."""
import numpy as np
import pytest

from tests import smallgraphs as sg

pytestmark = pytest.mark.gpu

N = 1104  # (2^30 - 2) / 1103 is a whole number, and searches beyond 1,024 vertices run in buckets
W = ((1 << 30) - 2) // (N - 1)


@pytest.fixture(scope="module")
def gcm():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1710_01144_gb300 import build, gc

    build.build()
    return gc


def test_path_of_largest_weights(gcm):
    assert W * (N - 1) == (1 << 30) - 2
    rp, ci = sg.path(N)
    with gcm.Graph(rp, ci) as G:
        want, f, _ = G.greedy(5)  # all weights equal: the unweighted groups
        G.set_weights(np.full(ci.size, W, np.int32), validate=True)
        got, fw, _ = G.greedy_weighted(5)
        np.testing.assert_array_equal(got, want)
        assert fw == W * f
        with pytest.raises(gcm.GcError) as e:
            G.set_weights(np.full(ci.size, W + 1, np.int32))
        assert e.value.code == gcm.GC_ERANGE


def test_pending_entry_at_the_largest_length(gcm):
    """From an end of a path of N - 1 vertices with one more vertex beside it, the
    last entry back leads to a length of exactly 2^30 - 2: the search must end and
    report the graph as disconnected."""
    rp, ci = sg.disjoint_union(sg.path(N - 1), sg.path(1))
    with gcm.Graph(rp, ci) as G:
        G.set_weights(np.full(ci.size, W, np.int32))
        with pytest.raises(gcm.GcError) as e:
            G.greedy_weighted(3)
        assert e.value.code == gcm.GC_EDISCONNECTED
