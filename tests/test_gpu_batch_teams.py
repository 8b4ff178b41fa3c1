"""The batched solver's lazy rounds by teams of CTAs: every team size, list
capacity and form of a step (shared-memory list, grid selection over every
candidate, wide steps on deep graphs) must give each graph's oracle group."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1710_01144_gb300 import graphgen
from tests import smallgraphs as sg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1710_01144_gb300 import build, gc

    build.build()
    graphs = [graphgen.barabasi_albert(700 + 311 * i, 1 + i, 3 + i) for i in range(4)]
    graphs += [graphgen.rmat(11, 3.0, seed=2), graphgen.rmat(13, 5.0, seed=6), sg.path(90), sg.cycle(61),
               graphgen.grid_road(40, 33, 0.2, 0.01, 4), sg.star(25), graphgen.rmat(9, 2.0, seed=8)]
    ks = [9, 21, 3, 14, 12, 30, 8, 5, 11, 4, 17]
    ref = [oracle.greedypp(rp, ci, k) for (rp, ci), k in zip(graphs, ks)]
    return gc, graphs, ks, [(r[0], int(r[1][-1])) for r in ref]


@pytest.mark.parametrize("team", [0, 1, 3, 16, 152, 1000])
@pytest.mark.parametrize("cap", [0, 2, 100, 5000])
def test_teams_match_oracle(env, team, cap):
    gc, graphs, ks, ref = env
    lib = gc.load()
    ksa = np.array(ks, dtype=np.int32)
    with gc.Batch(graphs) as B:
        for flags in (0, gc.GC_OPT_CAPTURE, gc.GC_OPT_NO_ROUND1_BOUND):
            o = gc.Opts()
            lib.gc_opts_default(ctypes.byref(o))
            o.lazy_ctas, o.active_target, o.flags = team, cap, flags
            groups, far = np.zeros(int(ksa.sum()), np.int32), np.zeros(len(ks), np.int64)
            gc._check(lib.gc_batch_greedy(B._h, ksa.ctypes.data, ctypes.byref(o), groups.ctypes.data,
                                          far.ctypes.data, None))
            at = 0
            for i, (k, (grp, f)) in enumerate(zip(ks, ref)):
                np.testing.assert_array_equal(groups[at:at + k], grp, err_msg="graph %d" % i)
                assert far[i] == f
                at += k
