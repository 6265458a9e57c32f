"""The FP32 block solves at the edges of their 32-row tiles and of the batches of rows that the
streaming warps keep in flight, in every launch shape and both groupings of right-hand sides."""
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


@pytest.fixture
def trsv():
    """Sets the launch shape of the block solves; automatic again afterwards."""
    from paper_1305_6653_gb300 import _lib
    yield lambda v: _lib.load().fde_tune_set(_lib.FDE_TUNE_TRSV, v)
    _lib.load().fde_tune_set(_lib.FDE_TUNE_TRSV, -1)


@pytest.mark.parametrize("m,s", [(3, 16), (64, 32), (65, 16), (128, 64), (190, 32), (257, 16), (449, 32), (770, 16),
                                 (1500, 16)])
def test_residual_in_every_launch_shape(trsv, m, s):
    """S z = r: factors of growth <= 2, tile inverses and two substitutions in FP32 leave a residual of
    at most about 12 (m + 32) u |S| |z|, the transforms in time 14 log2(s) u (|r| + |S| |z|)."""
    from paper_1305_6653_gb300 import FDEProblem
    prob = fi.manufactured(m, s, 1.4, "GBDF3", dplus_fn=lambda x: 1.0 + x, dminus_fn=lambda x: 2.0 - x)
    r = np.random.default_rng(m).standard_normal(prob.n)
    out = []
    with FDEProblem.from_inputs(prob, device_inputs=True) as p:
        p.assemble().factor("fp32")
        for v in range(4):
            trsv(v)
            out.append(p.precond_apply(torch.as_tensor(r, device="cuda")).cpu().numpy())
    for z in out[1:]:
        assert np.array_equal(z, out[0])
    z = out[0]
    phi, psi = O.strang_symbols(prob.family, prob.mu, s)
    jn = 2 * prob.alpha * (prob.dplus + prob.dminus).max() * prob.dx ** (-prob.alpha)
    sn = np.abs(phi).max() + prob.h * np.abs(psi).max() * jn
    u = 2.0 ** -24
    rn, zn = np.linalg.norm(r), np.linalg.norm(z)
    assert np.linalg.norm(O.strang_matvec(prob, z) - r) <= (12 * (m + 32) * u * sn * zn
                                                            + 14 * np.log2(s) * u * (rn + sn * zn))


@pytest.mark.parametrize("m,s,count", [(65, 256, 9), (129, 32, 5), (40, 16, 3), (300, 64, 17)])
def test_right_hand_sides_in_groups_of_four_and_eight(m, s, count):
    """129 blocks and 9 right-hand sides go in groups of 8, the others in groups of 4; full and short
    groups, each solution against the oracle's FP64 solve (both to 1e-11 of a well-conditioned system)."""
    from paper_1305_6653_gb300 import FDEBatch
    probs = fi.config_many_rhs(count=count, m=m, s=s)
    with FDEBatch(probs) as b:
        b.share_operator().block_solver("cuda_cores").assemble().factor("fp32")
        xs, stats = b.solve(tol=1e-11, restart=20, maxit=400)
        xs = [x.cpu().numpy() for x in xs]
    for i in {0, count // 2, count - 1}:
        ref, _, ok, _ = O.solve_strang_gmres(probs[i], side="right", tol=1e-11)
        assert ok and stats[i]["status"] == 0
        assert np.linalg.norm(xs[i] - ref) <= 1e-8 * np.linalg.norm(ref)
