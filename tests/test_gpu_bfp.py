"""The block floating-point space-time product at the sizes where it can go wrong: one and
two points, sizes beside the powers of two (each of its pass sequences), the largest m."""
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


@pytest.mark.parametrize("variant", [0, 2])
@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 8, 9, 16, 17, 33, 64, 65, 129, 257, 513, 1025, 2049, 4095])
def test_product_against_dense(m, variant):
    """Each entry within 64 units of FP64 rounding of sum |M_ij| |z_j| (the dense product's own
    rounding and two rounded FFTs are each below half of that); exactly homogeneous under powers
    of two, whose product shifts no integer of a row; a zero vector gives zeros."""
    from paper_1305_6653_gb300 import FDEProblem, _lib, fde_tune_set
    scheme = ("GBDF3", "GAM4", "ETR3", "GBDF5")[m % 4]
    prob = fi.manufactured(m, 16, 1.7, scheme, dplus_fn=lambda x: 1.0 + x, dminus_fn=lambda x: 2.0 - x)
    z = np.random.default_rng(m).standard_normal(prob.n)
    J = O.j_of(prob)
    A, B = O.bvm_matrices(prob.family, prob.mu, prob.s)
    ref = O.matvec(prob, z, J=J, AB=(A, B)).reshape(prob.s, m)
    Z = np.abs(z).reshape(prob.s, m)
    bound = np.abs(A[1:, 1:]) @ Z + prob.h * (np.abs(B[1:, 1:]) @ Z) @ np.abs(J).T
    fde_tune_set(_lib.FDE_TUNE_MATVEC, variant)
    try:
        with FDEProblem.from_inputs(prob, device_inputs=True) as p:
            p.assemble()
            zt = torch.as_tensor(z, device="cuda")
            y = p.matvec(zt)
            assert np.all(np.abs(y.cpu().numpy().reshape(prob.s, m) - ref) <=
                          64 * 2.0 ** -53 * bound.max(axis=1, keepdims=True))
            for k in (-600, 600):
                assert torch.equal(p.matvec(zt * 2.0 ** k), y * 2.0 ** k)
            assert torch.equal(p.matvec(torch.zeros_like(zt)), torch.zeros_like(zt))
    finally:
        fde_tune_set(_lib.FDE_TUNE_MATVEC, -1)


def test_non_finite_entries_spread_over_their_rows():
    """A NaN or infinity makes the rows non-finite whose band reaches it, and no other row."""
    from paper_1305_6653_gb300 import FDEProblem
    prob = fi.manufactured(63, 32, 1.5, "GBDF3")
    z = torch.ones(prob.n, dtype=torch.float64, device="cuda")
    for bad in (float("nan"), float("inf")):
        zb = z.clone()
        zb[20 * 63 + 7] = bad
        with FDEProblem.from_inputs(prob, device_inputs=True) as p:
            y = p.assemble().matvec(zb).reshape(32, 63)
        rows = ~torch.isfinite(y).all(dim=1)
        assert not torch.isfinite(y[20]).any()
        assert rows.sum() <= 2 * prob.mu + 1 and torch.isfinite(y[~rows]).all()
