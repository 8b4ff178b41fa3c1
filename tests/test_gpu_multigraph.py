"""Adjacencies that nobody validated: entries that repeat, entries of the vertex
itself, rows in any order.  Distances do not change, so neither do groups, gains
and farness values."""
import numpy as np
import pytest

import oracle
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


def _csr(n, src, dst, rng=None):
    order = np.lexsort((dst, src)) if rng is None else np.lexsort((rng.random(src.size), src))
    rp = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int32)
    return rp, dst[order].astype(np.int32)


def variants(rp, ci):
    n = rp.size - 1
    rng = np.random.default_rng(3)
    src, dst = np.repeat(np.arange(n), np.diff(rp)), ci.astype(np.int64)
    keep = src < dst
    u, v = src[keep], dst[keep]
    twice = rng.random(u.size) < 0.3
    uu, vv = np.concatenate([u, u[twice]]), np.concatenate([v, v[twice]])
    own = np.arange(n)
    yield "repeated", _csr(n, np.concatenate([uu, vv]), np.concatenate([vv, uu]))
    yield "repeated, any order", _csr(n, np.concatenate([uu, vv]), np.concatenate([vv, uu]), rng)
    yield "own vertex", _csr(n, np.concatenate([u, v, own]), np.concatenate([v, u, own]))
    yield "any order", _csr(n, src, dst, rng)


@pytest.mark.parametrize("name,g", [("ba", graphgen.barabasi_albert(300, 2, 1)), ("rmat", graphgen.rmat(10, 6.0, seed=2)),
                                    ("rmat12", graphgen.rmat(12, 5.0, seed=3)),
                                    ("road", graphgen.grid_road(20, 20, 0.2, 0.01, 5))])
def test_same_results(gcm, name, g):
    rp, ci = g
    n, k = rp.size - 1, 12
    grp, ft, _ = oracle.greedy_plain(rp, ci, k)
    S = grp[:2]
    ref = oracle.gains(rp, ci, S, np.arange(n))
    with gcm.Graph(rp, ci, validate=True) as G, gcm.Graph(rp, ci) as H:
        for x in (G, H):
            np.testing.assert_array_equal(x.greedy(k)[0], grp)
    for what, m in variants(rp, ci):
        with gcm.Graph(*m) as G:
            for kw in ({}, {"step_mode": 2}, {"claim_log": False}, {"pruned_adjacency": False}):
                got, f, _ = G.greedy(k, **kw)
                np.testing.assert_array_equal(got, grp, err_msg=what)
                assert f == ft[-1]
            np.testing.assert_array_equal(G.gains(S, np.arange(n)), ref, err_msg=what)
        with gcm.Batch([m, (rp, ci)]) as B:
            groups, far, _ = B.greedy([k, k])
            for q in groups:
                np.testing.assert_array_equal(q, grp, err_msg=what)
            assert far.tolist() == [ft[-1], ft[-1]]
