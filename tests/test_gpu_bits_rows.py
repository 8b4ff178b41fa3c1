"""bitGreedy++ in shared memory on rows around the lengths at which a thread, a warp
and several passes of a warp take them, several of them in one group of 32 vertices,
and targets whose rows hold one another.  Groups against gc_greedy."""
import numpy as np
import pytest

from paper_1710_01144_gb300 import graphgen

pytestmark = pytest.mark.gpu


def csr(n, u, v):
    key = np.unique(np.concatenate([u, v]).astype(np.int64) * n + np.concatenate([v, u]))
    src, dst = key // n, key % n
    rp = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))])
    return rp.astype(np.int32), dst.astype(np.int32)


def lattice(n, h):
    """A ring of n vertices, each joined to the h next ones: rows of 2 h."""
    u = np.repeat(np.arange(n), h)
    return csr(n, u, (u + np.tile(np.arange(1, h + 1), n)) % n)


def mixed(n, lengths, seed):
    """A random graph in which vertex v draws lengths[v % len(lengths)] neighbours."""
    r = np.random.default_rng(seed)
    u = np.repeat(np.arange(n), np.asarray(lengths)[np.arange(n) % len(lengths)])
    v = (u + r.integers(1, n, u.size)) % n
    tree = np.arange(1, n)
    return csr(n, np.concatenate([u, tree]), np.concatenate([v, (r.random(n - 1) * tree).astype(np.int64)]))


GRAPHS = [(f"lattice{n}x{h}", lattice(n, h)) for n, h in [(64, 3), (257, 4), (300, 8), (1000, 16), (1000, 17), (700, 33),
                                                          (2500, 64), (400, 160)]]
GRAPHS += [("mixed1", mixed(1500, [1, 1, 1, 200, 1, 1, 40], 1)), ("mixed2", mixed(3100, [2, 3, 5, 9, 17], 2)),
           ("mixed3", mixed(900, [60], 3)), ("mixed4", mixed(8200, [1, 12], 4)), ("complete90", csr(90, *np.triu_indices(90, 1)))]


@pytest.mark.parametrize("name,g", GRAPHS, ids=[x[0] for x in GRAPHS])
def test_rows(name, g):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1710_01144_gb300 import build, gc

    build.build()
    with gc.Graph(*g, validate=True) as G:
        want, f, _ = G.greedy(7)
        got, f2, _ = G.greedy_bits(7)
    np.testing.assert_array_equal(got, want)
    assert f == f2
