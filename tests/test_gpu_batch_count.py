"""Batches of thousands of instances: the count is no limit of a Gram-Schmidt step."""
import numpy as np
import pytest

import fde_inputs as fi
import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_more_instances_than_a_staged_step_has_room_for():
    """4,400 instances at a restart of 24, the largest stage of V in shared memory: many pieces of the
    list, most instances taken by one CTA alone, in the end a single one by all CTAs; the checked
    solutions against the oracle's direct solve as in the other batch tests."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1305_6653_gb300 import FDEBatch
    kinds = [fi.random_modes((3, 7, 12)[i % 3], (16, 32)[i % 2], ("GBDF3", "GAM4", "ETR3")[i % 3], 200 + i)
             for i in range(24)]
    kinds.append(fi.random_modes(60, 64, "ETR3", 7, alpha=1.9))  # converges last, alone
    probs = [kinds[i % 24] for i in range(4399)] + [kinds[24]]
    with FDEBatch(probs) as b:
        xs, stats = b.assemble().factor("fp32").solve(tol=1e-11, restart=24, maxit=400)
    assert all(st["status"] == 0 for st in stats)
    refs = [O.direct_solve(p) for p in kinds]
    for i in [*range(0, 4399, 37), 4399]:
        ref = refs[24 if i == 4399 else i % 24]
        assert np.linalg.norm(xs[i].numpy() - ref) <= 1e-8 * np.linalg.norm(ref)


def test_the_same_batch_gives_the_same_bits():
    """Twice over (the second time from captured cycles) and in a batch made anew: the same bits; alone
    the last bits may differ, the solution is the oracle's."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1305_6653_gb300 import FDEBatch
    probs = [fi.random_modes(m, s, sch, 31 + m) for m, s, sch in
             [(63, 32, "GBDF3"), (255, 64, "GAM4"), (31, 16, "ETR3"), (130, 128, "GBDF5")]]
    outs = []
    for _ in range(2):
        with FDEBatch(probs) as b:
            b.assemble().factor("fp32")
            for _ in range(2):
                outs.append([x.numpy().copy() for x in b.solve(tol=1e-11, restart=10, maxit=400)[0]])
    for xs in outs[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(xs, outs[0]))
    with FDEBatch(probs[2:3]) as b:
        alone = b.assemble().factor("fp32").solve(tol=1e-11, restart=10, maxit=400)[0][0].numpy()
    ref = O.direct_solve(probs[2])
    for x in (alone, outs[0][2]):
        assert np.linalg.norm(x - ref) <= 1e-8 * np.linalg.norm(ref)
