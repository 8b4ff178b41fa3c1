"""gc_set_weights: rows ordered by weight in one to four passes, rows on both sides of
the length from which a CTA sorts them, rows of one weight, weights set again on one
handle.  Weighted groups against the oracle on stars of stars."""
import numpy as np
import pytest

import oracle
from paper_1710_01144_gb300 import graphgen

pytestmark = pytest.mark.gpu


def hubs(leaves):
    """Hubs in a row with leaves[i] leaves each, the leaves of a hub in a ring of their own."""
    h = len(leaves)
    first = h + np.concatenate([[0], np.cumsum(leaves)])
    u, v = [np.arange(h - 1)], [np.arange(1, h)]
    for i, c in enumerate(leaves):
        x = first[i] + np.arange(c)
        u += [np.full(c, i), x[:-1]]
        v += [x, x[1:]]
    u, v, n = np.concatenate(u), np.concatenate(v), int(first[-1])
    key = np.unique(np.concatenate([u, v]).astype(np.int64) * n + np.concatenate([v, u]))
    src, dst = key // n, key % n
    rp = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))])
    return rp.astype(np.int32), dst.astype(np.int32)


@pytest.mark.parametrize("leaves", [[3, 40, 1], [2046, 2047], [2048, 3], [300, 2049, 31, 33]])
def test_rows_by_weight(leaves):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1710_01144_gb300 import build, gc

    build.build()
    rp, ci = hubs(leaves)
    n = rp.size - 1
    with gc.Graph(rp, ci) as G:
        for w_max in (1, 255, 256, 65535, 65536, min(2**24 + 5, (2**30 - 1) // n), 2):
            if w_max * (n - 1) >= 2**30:
                continue
            w = graphgen.edge_weights(rp, ci, w_max, 3)
            want, ft, _ = oracle.wgreedy_plain(rp, ci, w, 2)
            G.set_weights(w, validate=True)
            got, f, _ = G.greedy_weighted(2)
            np.testing.assert_array_equal(got, want)
            assert f == ft[-1]
