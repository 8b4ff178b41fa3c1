"""The one-source searches of deep graphs keep their queues in the workspaces of the
64-lane batches: a sparse handle takes no more memory than a dense one, and the
workspaces are zero again after every search."""
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


def _ring(n, half):
    """Every vertex joined to the `half` next ones on each side."""
    ci = (np.arange(n)[:, None] + np.concatenate([np.arange(-half, 0), np.arange(1, half + 1)])[None, :]) % n
    return (np.arange(n + 1) * 2 * half).astype(np.int32), np.sort(ci, axis=1).ravel().astype(np.int32)


def test_memory_of_a_sparse_handle(gcm):
    import torch

    n = 65536
    used = {}
    for half in (5, 1):  # ten neighbours (no one-source searches), two
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        with gcm.Graph(*_ring(n, half)):
            used[half] = before - torch.cuda.mem_get_info()[0]
    assert used[1] <= used[5]


@pytest.mark.parametrize("name,g", [("road64", graphgen.grid_road(64, 64, 0.2, 0.01, 2)), ("path4001", sg.path(4001)),
                                    ("grid3x333", sg.grid(3, 333))])
def test_batches_after_searches(gcm, name, g):
    import torch

    rp, ci = g
    n = rp.size - 1
    far = np.array([n // 2], np.int32)             # deep: one source per CTA
    near = np.arange(0, n, 5).astype(np.int32)     # shallow: 64-lane batches
    cand = np.arange(0, n, 3).astype(np.int32)
    ref = {1: oracle.gains(rp, ci, far, cand), 2: oracle.gains(rp, ci, near, cand)}
    out = torch.zeros(cand.size, dtype=torch.int64, device="cuda")
    dev = [torch.from_numpy(a).cuda() for a in (far, near, cand)]
    with gcm.Graph(rp, ci) as G:
        want, f, _ = G.greedy(4, round0_lanes=-1)  # the 64-lane form throughout
        ids, vals, _ = G.top_closeness(9, round0_lanes=-1)
        for _ in range(2):
            np.testing.assert_array_equal(G.gains(far, cand), ref[1])
            np.testing.assert_array_equal(G.gains(near, cand), ref[2])
            for i in (1, 2):
                G.gains_device(dev[i - 1], dev[2], out)
                np.testing.assert_array_equal(out.cpu().numpy(), ref[i])
            for kw in ({}, {"round0_lanes": -1}):
                got, f2, _ = G.greedy(4, **kw)
                np.testing.assert_array_equal(got, want)
                assert f == f2
                t, v, _ = G.top_closeness(9, **kw)
                np.testing.assert_array_equal(t, ids)
                np.testing.assert_array_equal(v, vals)
