"""Per-lane claim sums (warp_lane_sums in csrc/gc_device.cuh): claims of one and of
many lanes, weights of several bits (long distances), batches of 1 to 64 lanes, in
the CTA and the grid form, gains and farness."""
import numpy as np
import pytest

import oracle
from paper_1710_01144_gb300 import graphgen

pytestmark = pytest.mark.gpu


def _caterpillar(n, legs):
    """A path of n vertices with `legs` leaves at each: long distances, and
    leaves whose gains differ from lane to lane."""
    from scipy.sparse import coo_matrix

    a = np.arange(n - 1)
    leaf = n + np.arange(n * legs)
    e = np.concatenate([np.stack([a, a + 1]), np.stack([leaf, np.repeat(np.arange(n), legs)])], axis=1)
    m = n + n * legs
    c = coo_matrix((np.ones(2 * e.shape[1]), (np.concatenate([e[0], e[1]]), np.concatenate([e[1], e[0]]))),
                   shape=(m, m)).tocsr()
    c.sort_indices()
    return c.indptr.astype(np.int32), c.indices.astype(np.int32)


@pytest.mark.parametrize("lanes", [1, 31, 32, 33, 64])
@pytest.mark.parametrize("name", ["caterpillar", "ba"])
def test_sums(name, lanes):
    from paper_1710_01144_gb300 import build, gc

    build.build()
    rp, ci = _caterpillar(90, 3) if name == "caterpillar" else graphgen.barabasi_albert(300, 2, 5)
    n = rp.size - 1
    rng = np.random.default_rng(lanes)
    S = np.arange(0, n, max(1, n // 12), dtype=np.int32)[:12] if name == "ba" else np.arange(12, dtype=np.int32)
    cand = rng.choice(n, size=lanes, replace=False).astype(np.int32)
    with gc.Graph(rp, ci) as G:
        np.testing.assert_array_equal(G.gains(S, cand), oracle.gains(rp, ci, S, cand))
        want, ft = oracle.greedypp(rp, ci, 8)[:2]
        for kw in ({"step_mode": 2}, {"step_mode": 1, "eval_per_step": lanes, "step_lanes": lanes}, {"step_form": 1}):
            grp, f, _ = G.greedy(8, round0_lanes=-1, **kw)
            np.testing.assert_array_equal(grp, want)
            assert f == ft[-1]
        ids, far, _ = G.top_closeness(lanes, round0_lanes=-1)
        d = np.array([int(oracle.bfs(rp, ci, np.array([v], np.int32)).astype(np.int64).sum()) for v in range(n)])
        order = np.lexsort((np.arange(n), d))[:lanes]
        np.testing.assert_array_equal(ids, order)
        np.testing.assert_array_equal(far, d[order])
