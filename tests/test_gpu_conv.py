"""The network's convolutions at the edges of their tiles: images of odd numbers
of 4 x 4 cells (quarter-size images with odd widths, rows past a tile), channel
counts that fill no 16-, 32- or 64-channel tile, one sample and several, both
block sizes of each form.

Tolerances: a layer rounds each output by a few 2^-24 (products exact or fused,
sums in FP32), nine layers in a row: forward 2e-6 relative L2; the loss is a
mean over thousands of outputs, 1e-6; a gradient has up to nine such layers
behind it and a sum over the pixels of the batch: 1e-5 per layer."""
import numpy as np
import pytest

from oracle import warmnet as WN
from paper_1601_08201_gb300 import wsnet

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def case(H, W, Q, N, n_dual, seed):
    rng = np.random.default_rng(seed)
    net = wsnet.WarmNet(H, W, Q, max_batch=N, seed=seed, n_dual=n_dual)
    lay, _ = WN.layout(Q, n_dual)
    params = net.get_params()
    for w0, b0, ci, co in lay:
        params[b0:b0 + co] = 0.05 * rng.standard_normal(co)
    net.set_params(params)
    x = rng.random((N, Q + 1, H, W)).astype(np.float32)
    t = rng.random((N, Q * (1 + n_dual), H, W)).astype(np.float32)
    return net, params, x, t, lay


@pytest.mark.parametrize("H,W,Q,N,n_dual", [(4, 4, 1, 1, 0), (8, 12, 3, 2, 2), (12, 20, 17, 1, 0), (20, 36, 13, 3, 4),
                                            (36, 20, 37, 2, 1), (64, 64, 16, 1, 0), (32, 64, 15, 6, 0)])
def test_forward_loss_and_gradients(H, W, Q, N, n_dual):
    net, params, x, t, lay = case(H, W, Q, N, n_dual, seed=H + W + Q)
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    out = torch.empty_like(td)
    torch.cuda.synchronize()  # the network runs on its own stream
    net.forward(xd.data_ptr(), N, out.data_ptr())
    torch.cuda.synchronize()
    p64, x64 = params.astype(np.float64), x.astype(np.float64)
    ref = WN.forward(p64, x64, Q, n_dual=n_dual)
    assert np.linalg.norm(out.cpu().numpy() - ref) <= 2e-6 * np.linalg.norm(ref)
    loss = net.loss_grad(xd.data_ptr(), td.data_ptr(), N)
    g = net.get_grads().astype(np.float64)
    oloss, og = WN.loss_grad(p64, x64, t.astype(np.float64), Q, n_dual=n_dual)
    assert loss == pytest.approx(oloss, rel=1e-6)
    for l, (w0, b0, ci, co) in enumerate(lay):
        for a, b in ((g[w0:b0], og[w0:b0]), (g[b0:b0 + co], og[b0:b0 + co])):
            assert np.linalg.norm(a - b) <= 1e-5 * max(np.linalg.norm(b), 1e-12), l


def test_infinite_input_reaches_its_outputs_only():
    # nonnegative weights, so that no layer turns the infinity into a NaN that its ReLU drops: one infinite
    # pixel makes the outputs around it infinite and leaves those out of its reach as they were
    H = W = 64
    net, params, x, t, lay = case(H, W, 2, 1, 0, seed=5)
    net.set_params(np.abs(params))
    xd = torch.from_numpy(x).cuda()
    out, bad = torch.empty(1, 2, H, W, device="cuda"), torch.empty(1, 2, H, W, device="cuda")
    torch.cuda.synchronize()
    net.forward(xd.data_ptr(), 1, out.data_ptr())
    torch.cuda.synchronize()
    xd[0, 0, 0, 0] = float("inf")
    torch.cuda.synchronize()
    net.forward(xd.data_ptr(), 1, bad.data_ptr())
    torch.cuda.synchronize()
    assert torch.isfinite(out).all()
    assert torch.isposinf(bad[0, :, :4, :4]).all()
    assert torch.equal(bad[0, :, 48:, 48:], out[0, :, 48:, 48:])
