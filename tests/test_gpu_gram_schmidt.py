"""The Gram-Schmidt step in each of its forms: one element a thread in CTAs of 64, 128 and 256,
the loop over staged pairs and single elements, and the batched one with more instances than
SMs.  Plain GMRES over one cycle of 63 steps passes every register bucket."""
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


@pytest.mark.parametrize("reorth", [0, 1])
@pytest.mark.parametrize("m,s", [(9, 16), (63, 32), (255, 64), (511, 64), (333, 128), (1023, 64)])
def test_estimate_is_the_true_residual(m, s, reorth):
    """One cycle of k steps: the Givens estimate equals the recomputed residual norm if V is
    orthonormal, H is the projected operator and the rotations are right.  With re-orthogonalised
    FP64 vectors both carry errors of about k n^(1/2) 2^-53 < 1e-12 of |b|; a single pass loses
    orthogonality with the residual's decay, which plain GMRES has little of here."""
    from paper_1305_6653_gb300 import FDEProblem
    prob = fi.manufactured(m, s, 1.5, "GBDF3", dplus_fn=lambda x: 1.0 + x, dminus_fn=lambda x: 2.0 - x)
    with FDEProblem.from_inputs(prob, device_inputs=True) as p:
        p.assemble().no_precond()
        for k in (1, 2, 8, 9, 17, 25, 33, 63):
            x, st = p.solve(tol=1e-15, restart=k, maxit=k, reorth=reorth, raise_on_error=False)
            assert st["iterations"] == k
            assert abs(st["rel_residual"] - st["rel_residual_estimate"]) <= (1e-11 if reorth else 1e-7)


def test_batch_with_more_instances_than_sms():
    """160 small instances of uneven length: more than the 152 CTAs of a step, then fewer as
    they converge; every solution against the oracle's direct solve."""
    from paper_1305_6653_gb300 import FDEBatch
    probs = [fi.random_modes((7, 12, 20, 31)[i % 4], (16, 32)[i % 2], ("GBDF3", "GAM4", "ETR3")[i % 3], 100 + i)
             for i in range(160)]
    with FDEBatch(probs) as b:
        xs, stats = b.assemble().factor("fp32").solve(tol=1e-11, restart=10, maxit=400)
    for pr, x, st in list(zip(probs, xs, stats))[::9]:
        ref = O.direct_solve(pr)
        assert st["status"] == 0
        assert np.linalg.norm(x.numpy() - ref) <= 1e-8 * np.linalg.norm(ref), pr.name


@pytest.mark.parametrize("m,s,restart,maxit", [(63, 32, 20, 200), (63, 32, 3, 200), (255, 64, 5, 7), (40, 16, 1, 4)])
def test_step_queued_ahead_changes_nothing(m, s, restart, maxit):
    """The step queued behind the last one of a cycle must leave everything as it is: solutions
    and statistics with the profiler on (a step at a time, direct launches), without it (one step
    ahead) and from captured graphs are the same to the bit."""
    from paper_1305_6653_gb300 import FDEProblem
    prob = fi.manufactured(m, s, 1.5, "GBDF3")
    with FDEProblem.from_inputs(prob, device_inputs=True) as p:
        p.assemble().factor("fp64")
        out = []
        for prof in (True, False, False):
            p.profile(prof)
            out.append(p.solve(tol=1e-10, restart=restart, maxit=maxit, raise_on_error=False))
    for x, st in out[1:]:
        assert torch.equal(x, out[0][0])
        for key in ("status", "iterations", "restarts", "rel_residual", "rel_residual_estimate"):
            assert st[key] == out[0][1][key], key
