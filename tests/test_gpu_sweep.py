"""Lazy rounds whose candidate list cannot certify a pick: many bounds still
reach the best exact gain, and they are evaluated in one sweep of CTA batches
(gc_greedy) or by the graph's team (gc_batch_greedy).  Sparse graphs with long
tails, where the two-hop bounds are loose, need it; the group must stay the
oracle's."""
import numpy as np
import pytest

import oracle
from paper_1710_01144_gb300 import graphgen

pytestmark = pytest.mark.gpu


def cases():
    return [(graphgen.barabasi_albert(12000, 1, 3), 14), (graphgen.rmat(14, 2.0, seed=5), 20),
            (graphgen.rmat(15, 3.0, seed=9), 25), (graphgen.barabasi_albert(9000, 2, 7), 30)]


def test_sweeps_keep_the_group():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1710_01144_gb300 import build, gc

    build.build()
    swept, ref = 0, []
    for (rp, ci), k in cases():
        grp, ft, _, _ = oracle.greedypp(rp, ci, k)
        ref.append((grp, int(ft[-1])))
        with gc.Graph(rp, ci) as G:
            base = G.greedy(2)[2]["gain64_launches"]  # rounds 0 and 1
            for target in (0, 64, 700):
                got, f, st = G.greedy(k, active_target=target, step_form=1)
                np.testing.assert_array_equal(got, grp)
                assert f == ft[-1]
                swept += st["gain64_launches"] - base
    assert swept > 0
    with gc.Batch([g for g, _ in cases()]) as B:
        for target in (0, 32):
            groups, far, _ = B.greedy([k for _, k in cases()], active_target=target)
            for got, f, (grp, fr) in zip(groups, far, ref):
                np.testing.assert_array_equal(got, grp)
                assert f == fr
