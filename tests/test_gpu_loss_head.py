"""The loss head of the training step alone: with all weights 0 the output is
softplus(0) on the image channels and 0 on the dual ones, the loss the mean of the
squared differences from the targets, and the last layer's bias gradient its
derivative summed over a channel's pixels. Planes of one element a thread and of
several pieces, few and many of them, pieces that end inside a block's round.

Tolerances: the differences are single FP32 subtractions, the squares and their sum
FP64: 1e-12. A bias gradient adds up to some thousand FP32 terms of mixed signs in
FP32: 1e-5 of the sum of their magnitudes."""
import numpy as np
import pytest

from paper_1601_08201_gb300 import wsnet

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def zero_net(H, W, Q, N, n_dual):
    net = wsnet.WarmNet(H, W, Q, max_batch=N, n_dual=n_dual)
    net.set_params(np.zeros(net.num_params, np.float32))
    x = torch.zeros(N, Q + 1, H, W, device="cuda")
    out = torch.empty(N, Q * (1 + n_dual), H, W, device="cuda")
    torch.cuda.synchronize()  # the network runs on its own stream
    net.forward(x.data_ptr(), N, out.data_ptr())
    torch.cuda.synchronize()
    return net, x, out


@pytest.mark.parametrize("H,W,Q,N,n_dual", [(4, 4, 1, 1, 0), (32, 32, 1, 1, 0), (36, 60, 1, 1, 2), (64, 64, 5, 3, 4),
                                            (128, 132, 2, 1, 1), (256, 256, 1, 1, 0), (8, 8, 64, 8, 4)])
def test_loss_and_its_derivative(H, W, Q, N, n_dual):
    net, x, out = zero_net(H, W, Q, N, n_dual)
    C = Q * (1 + n_dual)
    t = np.random.default_rng(H + W + C).standard_normal((N, C, H, W)).astype(np.float32)
    td = torch.from_numpy(t).cuda()
    torch.cuda.synchronize()
    loss = net.loss_grad(x.data_ptr(), td.data_ptr(), N)
    diff = out.cpu().numpy() - t
    assert loss == pytest.approx(np.mean(diff.astype(np.float64) ** 2), rel=1e-12)
    dz = 2.0 * diff.astype(np.float64) / diff.size
    dz[:, :Q] *= 0.5  # the derivative of softplus at 0
    db = net.get_grads()[-C:].astype(np.float64)
    assert (np.abs(db - dz.sum((0, 2, 3))) <= 1e-5 * np.abs(dz).sum((0, 2, 3))).all()


@pytest.mark.parametrize("size", [1e-39, 3e-45, 1e-38, 1e-37])
def test_differences_below_the_normal_range_count(size):
    net, x, out = zero_net(8, 12, 3, 2, 2)
    t = out.clone()
    t[:, 3:] = size
    torch.cuda.synchronize()
    loss = net.loss_grad(x.data_ptr(), t.data_ptr(), 2)
    d = float(np.float32(size))
    assert d > 0 and abs(loss / (d * d * 2 / 3) - 1) <= 1e-12


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_infinite_and_nan_targets_show_in_the_loss(bad):
    net, x, out = zero_net(8, 12, 3, 1, 0)
    t = out.clone()
    t[0, 1, 5, 7] = bad
    torch.cuda.synchronize()
    loss = net.loss_grad(x.data_ptr(), t.data_ptr(), 1)
    assert np.isnan(loss) if np.isnan(bad) else np.isposinf(loss)
