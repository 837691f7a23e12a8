"""The network on a batch of more rows than a grid's y dimension has tiles for
(65535 x 32): rows are independent, so the first and last of them equal the
same rows in a small batch bit for bit, and the loss is that of the outputs."""
import numpy as np
import pytest

from paper_1508_02766_gb300 import kde

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_more_rows_than_tiles_along_y():
    B = 65535 * 32 + 100
    net = kde.MLP(in_dim=64, hidden=128, out_dim=3, max_batch=B, seed=5)
    small = kde.MLP(in_dim=64, hidden=128, out_dim=3, max_batch=256, seed=5)
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn(B, 64, device="cuda", generator=g)
    T = torch.randn(B, 3, device="cuda", generator=g)
    Y = net.forward(X)
    for sl in (slice(0, 256), slice(B - 256, B)):
        assert torch.equal(Y[sl], small.forward(X[sl].contiguous()))
    loss = torch.empty(1, device="cuda")
    grads = torch.empty(net.nparam, device="cuda")
    net.loss_grad(X, T, loss=loss, grads=grads)
    ref = ((Y.double() - T.double()) ** 2).sum().item() / B
    # FP32 differences summed in FP64
    assert abs(loss.item() - ref) < 1e-5 * ref
    assert np.isfinite(grads.cpu().numpy()).all()
    net.check()
