"""Steps of the weighted searches that one warp takes alone: frontiers of 31 to 64
vertices, steps of up to 128 entries and beyond, rows that grow and shrink between
them, and dense rows taken by the whole CTA.  Groups against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1710_01144_gb300 import graphgen
from tests import smallgraphs as sg

pytestmark = pytest.mark.gpu


def csr(n, u, v):
    key = np.unique(np.concatenate([u, v]).astype(np.int64) * n + np.concatenate([v, u]))
    src, dst = key // n, key % n
    rp = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))])
    return rp.astype(np.int32), dst.astype(np.int32)


def spider(arms, length, leaves):
    """A centre with `arms` paths of `length` vertices, each with `leaves` leaves."""
    body = 1 + np.arange(arms * length)
    prev = np.where((body - 1) % length == 0, 0, body - 1)
    n = 1 + body.size
    leaf = n + np.arange(body.size * leaves)
    return csr(n + leaf.size, np.concatenate([body, leaf]), np.concatenate([prev, np.repeat(body, leaves)]))


GRAPHS = [(f"spider{a}x{l}+{f}", spider(a, l, f)) for a, l, f in
          [(1, 40, 0), (31, 12, 0), (32, 12, 0), (33, 12, 0), (64, 6, 0), (32, 9, 2), (32, 9, 3), (3, 40, 41), (2, 40, 63)]]
GRAPHS += [("path700", sg.path(700)), ("strip4x150", graphgen.grid_road(4, 150, 0.0, 0.0, 1)),
           ("complete150", csr(150, *np.triu_indices(150, 1))), ("path1200", sg.path(1200))]


@pytest.mark.parametrize("w_max", [1, 9, 700])
@pytest.mark.parametrize("name,g", GRAPHS, ids=[x[0] for x in GRAPHS])
def test_groups_match_oracle(name, g, w_max):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1710_01144_gb300 import build, gc

    build.build()
    rp, ci = g
    w = graphgen.edge_weights(rp, ci, w_max, 5)
    want, ft, _ = oracle.wgreedy_plain(rp, ci, w, 5)
    with gc.Graph(rp, ci) as G:
        G.set_weights(w, validate=True)
        for _ in range(2):  # the workspaces are at rest again
            got, f, _ = G.greedy_weighted(5)
            np.testing.assert_array_equal(got, want)
            assert f == ft[-1]
