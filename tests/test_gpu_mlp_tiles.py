"""Row tiles of the proposal network: remainders of both tile sizes, one row, the
line between them and several tiles a CTA, against the float64 reference."""
import numpy as np
import pytest

from oracle import mlp as mref

pytestmark = pytest.mark.gpu


def _net(max_batch):
    from paper_1710_01144_gb300 import build, gc

    build.build()
    net = gc.Mlp(max_batch=max_batch)
    net.set_params(mref.init_params(4).astype(np.float32))
    return net


def _slots():
    import torch

    return 2 * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("rows", [1, 15, 16, 17, "16s", "16s+1", "64s+5", "130s+63"])
def test_scores_and_gradient(rows):
    import torch

    if isinstance(rows, str):
        f, _, d = rows.partition("s")
        rows = int(f) * _slots() + int(d or 0)
    net = _net(rows)
    p = net.get_params().astype(np.float64)
    rng = np.random.default_rng(rows)
    # an offset of one float: rows without 16-byte alignment
    X = torch.from_numpy(rng.normal(size=rows * 8 + 1).astype(np.float32)).cuda()[1:].view(rows, 8)
    y = torch.from_numpy(rng.normal(size=rows + 1).astype(np.float32)).cuda()[1:]
    out = torch.full((rows + 1,), -7.0, dtype=torch.float32, device="cuda")
    net.forward(X, out[:rows])
    g, loss = net.grad(X, y)
    again, loss2 = net.grad(X, y)
    assert np.array_equal(g, again) and loss == loss2  # sums in a fixed order
    Xh, yh = X.cpu().numpy().astype(np.float64), y.cpu().numpy().astype(np.float64)
    got = out.cpu().numpy()
    assert got[rows] == -7.0
    np.testing.assert_allclose(got[:rows], mref.forward(p, Xh), rtol=1e-4, atol=1e-4)
    gref = mref.grad(p, Xh, yh)
    assert abs(loss - mref.loss(p, Xh, yh)) <= 1e-4 * max(1.0, abs(loss))
    o = 0
    for _, shape in mref.SIZES:
        k = int(np.prod(shape))
        scale = np.abs(gref[o:o + k]).max() + 1e-12
        np.testing.assert_allclose(g[o:o + k], gref[o:o + k], rtol=1e-3, atol=2e-5 * scale)
        o += k
    net.close()
