"""Deep graphs: one-source-per-CTA searches and the bounds they pass to their
neighbourhoods (csrc/gc_solo.cu).  Gains (host and device form), the greedy and
top-k closeness against the oracle, at the sizes where the kernel can go wrong:
bitmap words and 16-byte units, rows longer than a warp, more candidates than
CTAs, members, repeats and ids out of range."""
import numpy as np
import pytest

import oracle
from paper_1710_01144_gb300 import graphgen
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


def broom(length, leaves):
    """A path whose last vertex has many leaves: deep, with one long row."""
    n = length + leaves
    u = list(range(length - 1)) + [length - 1] * leaves
    v = list(range(1, length)) + list(range(length, n))
    src, dst = np.array(u + v), np.array(v + u)
    o = np.lexsort((dst, src))
    rp = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int32)
    return rp, dst[o].astype(np.int32)


def deep_cases():
    return [("path33", sg.path(33)), ("path127", sg.path(127)), ("path129", sg.path(129)), ("cycle512", sg.cycle(512)),
            ("grid3x40", sg.grid(3, 40)), ("broom", broom(70, 301)), ("road20", graphgen.grid_road(20, 61, 0.2, 0.01, 5)),
            ("road64", graphgen.grid_road(64, 64, 0.2, 0.01, 2)), ("cater", sg.caterpillar(60, 9))]


@pytest.mark.parametrize("name,g", deep_cases())
def test_gains(gcm, name, g):
    import torch

    rp, ci = g
    n = rp.size - 1
    rng = np.random.default_rng(4)
    with gcm.Graph(rp, ci) as G:
        for s in (1, 2):
            S = rng.choice(n, s, replace=False).astype(np.int32)
            cand = np.concatenate([np.arange(n), S, rng.integers(0, n, 2700 if n > 900 else 70)]).astype(np.int32)
            ref = oracle.gains(rp, ci, S, cand)
            np.testing.assert_array_equal(G.gains(S, cand), ref)
            Sd, cd = torch.from_numpy(S).cuda(), torch.from_numpy(np.append(cand, [-1, n]).astype(np.int32)).cuda()
            out = torch.zeros(cd.numel(), dtype=torch.int64, device="cuda")
            G.gains_device(Sd, cd, out)
            np.testing.assert_array_equal(out.cpu().numpy()[:-2], ref)
            assert out.cpu().numpy()[-2:].tolist() == [-1, -1]
            assert G.farness(S) == oracle.farness(rp, ci, S)  # the handle is as before


@pytest.mark.parametrize("name,g", deep_cases())
def test_greedy_and_top_closeness(gcm, name, g):
    rp, ci = g
    n = rp.size - 1
    k = min(n, 15)
    grp, ft, _ = oracle.greedy_plain(rp, ci, k)
    ids, far, _ = oracle.topk_closeness(rp, ci, k)
    with gcm.Graph(rp, ci) as G:
        for kk in (k, 1, 2):
            got, f, st = G.greedy(kk)
            np.testing.assert_array_equal(got, grp[:kk])
            assert f == ft[kk - 1]
        ti, tf, _ = G.top_closeness(k)
        np.testing.assert_array_equal(ti, ids)
        np.testing.assert_array_equal(tf, far)


@pytest.mark.parametrize("side,k", [(110, 12), (150, 6)])
def test_sampled_stages(gcm, side, k):
    """More candidates than two waves of CTAs: sampled stages and relaxed
    pruning; the group and every vertex's farness rank must stay the oracle's."""
    rp, ci = graphgen.grid_road(side, side, 0.2, 0.01, 7)
    grp, ft, _, _ = oracle.greedypp(rp, ci, k)
    with gcm.Graph(rp, ci) as G:
        got, f, st = G.greedy(k)
        np.testing.assert_array_equal(got, grp)
        assert f == ft[-1]
        assert st["evals"] < (k - 1) * (rp.size - 1)
        ids, far, _ = G.top_closeness(40)
        ids0, far0, _ = G.top_closeness(40, round0_lanes=-1)
        np.testing.assert_array_equal(ids, ids0)
        np.testing.assert_array_equal(far, far0)
