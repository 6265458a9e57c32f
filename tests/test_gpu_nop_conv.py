"""The network's convolutions where their tiles can go wrong: one mode, tiles that cross
samples, a ragged last tile, more channels than a chunk, the wide tile of large launches."""
import numpy as np
import pytest

from oracle import nop_oracle as N

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("s,modes,width,layers,K,B", [
    (2, 1, 3, 2, 7, 5), (3, 5, 17, 2, 3, 7), (16, 16, 64, 3, 5, 32), (70, 13, 16, 2, 1, 9), (33, 65, 40, 2, 7, 2),
    (5, 130, 64, 2, 5, 40), (150, 8, 200, 2, 3, 130)])
def test_forward_and_gradients(s, modes, width, layers, K, B):
    """Forward and every gradient against the FP64 oracle.  An FP32 sum of n products is within
    n 2^-24 of the sum of their magnitudes; with the networks' 2 to 3 layers and n <= 5,200
    terms of random sign (whose sum is about sqrt(n) of n terms) 1e-4 of the largest entry is
    a safe bound on every one."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1305_6653_gb300 import FDENop
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
