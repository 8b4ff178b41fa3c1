"""Row-window passes (csrc/gc_rows.cu): every window width, rows on both sides of
the long-row limit (2048), empty pruned rows, distances beyond the 4-bit classes,
against the two-hop bounds restated from the CSR and against the full adjacency."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gcm():
    from paper_1710_01144_gb300 import build, gc

    build.build()
    return gc


def _graph(n, hubs, tail, seed):
    """A random tree-like graph with hubs of about the long-row limit and a path of
    `tail` vertices at its end."""
    rng = np.random.default_rng(seed)
    m = n - tail
    parent = (np.arange(1, m) * rng.random(m - 1)).astype(np.int64)
    e = [np.stack([np.arange(1, m), parent])]
    e.append(rng.integers(0, m, size=(2, m)))
    for h, deg in enumerate(hubs):
        e.append(np.stack([np.full(deg, (h * 17) % m), rng.choice(m, size=deg, replace=False)]))
    e.append(np.stack([np.arange(m - 1, n - 1), np.arange(m, n)]))
    e = np.concatenate(e, axis=1)
    e = e[:, e[0] != e[1]]
    key = np.unique(np.concatenate([e[0] * n + e[1], e[1] * n + e[0]]))
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(key // n, minlength=n), out=rp[1:])
    return rp.astype(np.int32), (key % n).astype(np.int32)


def _dist(rp, ci, S):
    d = np.full(rp.size - 1, -1, dtype=np.int64)
    d[S] = 0
    src = np.repeat(np.arange(rp.size - 1), np.diff(rp))
    lev = 0
    while True:
        hit = ci[d[src] == lev]
        hit = hit[d[hit] < 0]
        if hit.size == 0:
            return d
        lev += 1
        d[hit] = lev


def _bound(rp, ci, d):
    n = rp.size - 1
    src = np.repeat(np.arange(n), np.diff(rp))
    c3 = np.bincount(src, weights=d[ci] >= 3, minlength=n).astype(np.int64)
    term = np.where(d >= 2, d - 1 + c3, 0)
    ub = d + np.bincount(src, weights=term[ci].astype(np.float64), minlength=n).astype(np.int64) + np.maximum(d - 3, 0).sum()
    ub[d == 0] = -1
    return ub


# widths of 1, 2, 4, 8, 16 and 32 rows on 152 SMs begin at 0, 38.9k, 77.8k, 156k, 311k and 622k vertices
@pytest.mark.parametrize("n", [2, 33, 700, 39000, 80001, 160000, 312003, 650001])
def test_bounds_and_groups(gcm, n):
    hubs = [d for d in (2047, 2048, 2049, 2060, 9000, 30000) if 8 * d < n]
    tail = 20 if n > 100 else 0
    rp, ci = _graph(n, hubs, tail, n)
    assert not hubs or np.diff(rp).max() > 2048
    with gcm.Graph(rp, ci) as G:
        for S in ([0], [n - 1], [0, n // 2, n - 1]):
            S = sorted(set(S))
            d = _dist(rp, ci, np.array(S))
            assert (d >= 0).all()
            np.testing.assert_array_equal(G.upper_bounds(S), _bound(rp, ci, d))
        k = min(n, 6)
        a, fa, _ = G.greedy(k)
        b, fb, _ = G.greedy(k, pruned_adjacency=False, expand_bound=False, r0_probe=False)
        np.testing.assert_array_equal(a, b)
        assert fa == fb
        ids, far, _ = G.top_closeness(3 if n > 2 else 1)
        v = int(ids[0])
        assert int(far[0]) == int(_dist(rp, ci, np.array([v])).sum())
        assert int(a[0]) == v
