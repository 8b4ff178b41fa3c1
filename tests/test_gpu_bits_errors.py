"""bitGreedy++ on a graph of many components: refused after round 0, whatever k."""
import time

import numpy as np
import pytest

from paper_1710_01144_gb300 import graphgen

pytestmark = pytest.mark.gpu


def test_disconnected_is_refused_at_once():
    import torch

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1710_01144_gb300 import build, gc

    build.build()
    rp, ci = graphgen.barabasi_albert(64, 2, 1)
    parts, n = 64, 64 * 64
    rps = np.concatenate([[0], (rp[1:][None, :] + ci.size * np.arange(parts)[:, None]).ravel()]).astype(np.int32)
    cis = (ci[None, :] + 64 * np.arange(parts)[:, None]).ravel().astype(np.int32)
    whole = graphgen.barabasi_albert(n, 2, 1)
    with gc.Graph(rps, cis) as G, gc.Graph(*whole) as H:
        want = H.greedy(5)[0]
        for k in (1, 2, 400, 400):
            torch.cuda.synchronize()
            t = time.perf_counter()
            with pytest.raises(gc.GcError) as e:
                G.greedy_bits(k)
            # 5 ms a round where every round sweeps all levels; 5 us a round to enqueue it
            assert time.perf_counter() - t < 0.2
            assert e.value.code == gc.GC_EDISCONNECTED
            np.testing.assert_array_equal(H.greedy_bits(5)[0], want)
        assert G.farness(np.arange(0, n, 1)) == 0  # the handle is usable
