"""Bias gradients of the network: their rounding, and that they repeat to the bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("s,modes,B", [(20, 1, 5), (3, 3, 17), (20, 16, 32), (1, 4095, 1), (17, 130, 33), (4, 1023, 64)])
def test_rounding_and_repeatability(s, modes, B):
    """One layer of zero weights, so the loss gradient of an output is -2 t / N rounded to FP32; all
    terms of a channel are equal, whose rounding errors add up in a long chain.  Sums of four in
    FP32, the rest in FP64: at most 3 units of 2^-24 of the sum of magnitudes and the final rounding."""
    from paper_1305_6653_gb300 import FDENop
    net = FDENop(max(modes, 7), s, modes=modes, width=8, layers=1, ksize=3)
    net.set_params(np.zeros(net.nparam, np.float32))
    t = np.broadcast_to(((np.arange(s) + 1) / np.float32(3)).astype(np.float32)[None, :, None], (B, s, modes))
    N = B * s * modes
    g = (2.0 * (np.float32(0) - t).astype(np.float32) * (1.0 / N)).astype(np.float32).astype(np.float64)
    want, mag = g.sum(axis=(0, 2)), np.abs(g).sum(axis=(0, 2))
    x = torch.randn(B * net.cin * modes, device="cuda", generator=torch.Generator("cuda").manual_seed(s))
    td = torch.as_tensor(np.ascontiguousarray(t).reshape(-1), device="cuda")
    _, grad = net.loss_grad(x, td, B, want_grad=True)
    assert np.all(np.abs(grad[-s:] - want) <= 2.0 ** -24 * (3 * mag + np.abs(want)))
    # two layers and random data: the same bits each time
    net = FDENop(max(modes, 7), s, modes=modes, width=24, layers=2, ksize=5, seed=s)
    rng = np.random.default_rng(s)
    net.set_params((0.1 * rng.standard_normal(net.nparam)).astype(np.float32))
    td = torch.as_tensor(rng.standard_normal(N).astype(np.float32), device="cuda")
    w0 = 24 * net.cin * 5
    biases = np.r_[w0:w0 + 24, net.nparam - s:net.nparam]
    first = net.loss_grad(x, td, B, want_grad=True)[1][biases]
    for _ in range(4):
        assert np.array_equal(net.loss_grad(x, td, B, want_grad=True)[1][biases], first)
