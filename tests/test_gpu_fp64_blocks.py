"""FP64 Strang blocks at the edges of their 32-row tiles, of the padding to 64, of the time
transform's tile widths and of the two block solves (up to 512 rows and beyond)."""
import numpy as np
import pytest

import fde_inputs as fi
import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


@pytest.mark.parametrize("m,s,scheme", [(1, 16, "GBDF3"), (2, 32, "ETR3"), (31, 32, "GBDF3"), (32, 16, "GAM4"),
                                        (33, 64, "GBDF5"), (63, 32, "GBDF3"), (64, 256, "GBDF3"), (65, 32, "GBDF3"),
                                        (96, 128, "GBDF3"), (97, 32, "ETR3"), (300, 16, "GBDF3"), (511, 32, "GAM4"),
                                        (512, 16, "GBDF3"), (513, 16, "GBDF3"), (600, 16, "GBDF3"), (961, 16, "ETR3")])
def test_residual_of_the_preconditioner_solve(m, s, scheme):
    """S z = r: an LU without pivoting of growth <= 2 (the blocks are diagonally dominant), the tile
    inverses and two substitutions leave a residual of at most about 12 (m + 32) u |S| |z|; the
    two transforms in time add 14 log2(s) u (|r| + |S| |z|)."""
    from paper_1305_6653_gb300 import FDEProblem
    prob = fi.manufactured(m, s, 1.4, scheme, dplus_fn=lambda x: 1.0 + x, dminus_fn=lambda x: 2.0 - x)
    r = np.random.default_rng(m).standard_normal(prob.n)
    with FDEProblem.from_inputs(prob, device_inputs=True) as p:
        z = p.assemble().factor("fp64").precond_apply(torch.as_tensor(r, device="cuda")).cpu().numpy()
    res = np.linalg.norm(O.strang_matvec(prob, z) - r)
    phi, psi = O.strang_symbols(prob.family, prob.mu, s)
    jn = 2 * prob.alpha * (prob.dplus + prob.dminus).max() * prob.dx ** (-prob.alpha)
    sn = np.abs(phi).max() + prob.h * np.abs(psi).max() * jn
    u = 2.0 ** -53
    rn, zn = np.linalg.norm(r), np.linalg.norm(z)
    assert res <= 12 * (m + 32) * u * sn * zn + 14 * np.log2(s) * u * (rn + sn * zn)
