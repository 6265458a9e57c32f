"""The network on a batch whose input passes 2^31 entries: offsets into it need 64 bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_batch_of_more_than_2_31_entries():
    """All samples are zero but the first and the last, which are equal: equal outputs to the bit
    (a position's sum does not depend on its tile), and a first-layer weight gradient that is
    1 / 256 of that of the two alone (the mean is over 256 times as many entries, a power of two)
    up to the rounding of FP32 sums, 1e-4 of the largest entry as in the other network tests."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1305_6653_gb300 import FDENop
    s, m, B, width, K = 1024, 4095, 512, 4, 3
    net = FDENop(m, s, modes=m, width=width, layers=2, ksize=K)
    assert (B - 1) * net.cin * m > 2 ** 31
    rng = np.random.default_rng(31)
    net.set_params((0.1 * rng.standard_normal(net.nparam)).astype(np.float32))
    one = torch.as_tensor(rng.standard_normal((net.cin, m)).astype(np.float32), device="cuda")
    two = torch.stack([one, one])
    x = torch.zeros((B, net.cin, m), dtype=torch.float32, device="cuda")
    x[0] = one
    x[-1] = one
    y = net.forward(x, B).reshape(B, s, m)
    y2 = net.forward(two, 2).reshape(2, s, m)
    assert torch.equal(y[-1], y[0]) and not torch.equal(y[1], y[0])
    assert (y[0] - y2[0]).abs().max() <= 1e-4 * y2.abs().max()
    del y
    _, g = net.loss_grad(x, torch.zeros((B, s, m), dtype=torch.float32, device="cuda"), B, want_grad=True)
    _, g2 = net.loss_grad(two, torch.zeros((2, s, m), dtype=torch.float32, device="cuda"), 2, want_grad=True)
    n = width * net.cin * K
    assert np.abs(256 * g[:n] - g2[:n]).max() <= 1e-4 * np.abs(g2[:n]).max()
    net.close()
    del x
    torch.cuda.empty_cache()
