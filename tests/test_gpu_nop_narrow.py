"""The network's convolutions with few input channels and many positions, whose warps take
positions of their own: ragged last tiles, tiles that cross samples, one mode, every kernel size."""
import numpy as np
import pytest

from oracle import nop_oracle as N

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("s,modes,width,layers,K,B", [(1, 2047, 16, 3, 7, 10), (2, 701, 5, 2, 1, 29),
                                                      (9, 1, 16, 2, 5, 19500), (10, 1300, 16, 2, 3, 16),
                                                      (3, 37, 33, 3, 3, 600)])
def test_forward_and_gradients(s, modes, width, layers, K, B):
    """Forward and every gradient against the FP64 oracle.  An FP32 sum of n products of random sign
    is off by about n^(1/2) 2^-24 of its terms' size times its length's root; the weight gradients are
    the longest, n = 22,200 positions in 16 chains of which each adds at most n / 16 terms: 1e-4 of
    the largest entry, as in the other network tests."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1305_6653_gb300 import FDENop
    assert B * modes >= 128 * 152
    net = FDENop(max(modes, 7), s, modes=modes, width=width, layers=layers, ksize=K, seed=1)
    shapes = N.layer_shapes(cin=s + 6, cout=s, width=width, layers=layers, K=K)
    rng = np.random.default_rng(s)
    theta = (rng.standard_normal(net.nparam) / np.sqrt(width * K)).astype(np.float32)
    net.set_params(theta)
    x = rng.standard_normal((B, net.cin, modes)).astype(np.float32)
    t = rng.standard_normal((B, s, modes)).astype(np.float32)
    xd, td = (torch.as_tensor(v.reshape(-1), device="cuda") for v in (x, t))
    y = net.forward(xd, B).cpu().numpy().reshape(B, s, modes)
    ref = N.forward(theta, shapes, x)
    assert np.abs(y - ref).max() <= 1e-4 * np.abs(ref).max()
    loss, g = net.loss_grad(xd, td, B, want_grad=True)
    loss_ref, g_ref = N.loss_and_grad(theta, shapes, x, t)
    assert abs(loss - loss_ref) <= 1e-5 * loss_ref
    o = 0
    for ci, co, k in shapes:  # weights and biases of each layer on their own scale
        for n in (co * ci * k, co):
            assert np.abs(g[o:o + n] - g_ref[o:o + n]).max() <= 1e-4 * np.abs(g_ref[o:o + n]).max()
            o += n
