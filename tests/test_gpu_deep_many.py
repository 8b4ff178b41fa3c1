"""Gains of many candidates on deep graphs: around the numbers of candidates and
vertices from which the first searches decide who takes the rest, on graphs where
either form does, through host and device arrays, twice on one handle and with more
candidates than vertices.  Against the 128-lane batches."""
import numpy as np
import pytest

from paper_1710_01144_gb300 import graphgen

pytestmark = pytest.mark.gpu


def with_tail(g, length):
    n = g[0].size - 1
    u = np.repeat(np.arange(n), np.diff(g[0]))
    p = np.concatenate([[0], n + np.arange(length)])
    u, v = np.concatenate([u, p[:-1], p[1:]]), np.concatenate([g[1], p[1:], p[:-1]])
    at = np.lexsort((v, u))
    rp = np.concatenate([[0], np.cumsum(np.bincount(u, minlength=n + length))])
    return rp.astype(np.int32), v[at].astype(np.int32)


GRAPHS = [("tail65535", with_tail(graphgen.barabasi_albert(65505, 2, 1), 30)),
          ("tail65536", with_tail(graphgen.barabasi_albert(65506, 2, 1), 30)),
          ("tail70000", with_tail(graphgen.barabasi_albert(70000, 3, 2), 20)),
          ("road280", graphgen.grid_road(280, 280, 0.2, 0.01, 3)), ("shallow", graphgen.barabasi_albert(70000, 3, 2))]


@pytest.mark.parametrize("name,g", GRAPHS, ids=[x[0] for x in GRAPHS])
def test_many_candidates(name, g):
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1710_01144_gb300 import build, gc

    build.build()
    n = g[0].size - 1
    rng = np.random.default_rng(3)
    with gc.Graph(*g) as G, gc.Graph(*g) as H:
        H.set_gain_lanes(128)
        for s, m in [(1, 32768), (1, 32769), (3, n), (40, n), (1, n + 40000)]:
            S = rng.choice(n, s, replace=False).astype(np.int32)
            c = rng.integers(0, n, m).astype(np.int32) if m != n else np.arange(n, dtype=np.int32)
            want = H.gains(S, c)
            np.testing.assert_array_equal(G.gains(S, c), want)
            if m <= n:
                out = torch.full((m,), -7, dtype=torch.int64, device="cuda")
                G.gains_device(torch.tensor(S, device="cuda"), torch.tensor(c, device="cuda"), out)
                np.testing.assert_array_equal(out.cpu().numpy(), want)
