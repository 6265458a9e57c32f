"""The factorisation of a batch is a fixed number of launches, whatever the number of instances."""
import pytest

import fde_inputs as fi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision,storage", [("fp32", "fp32"), ("tf32", "fp32"), ("tf32", "bf16")])
def test_factorisation_launches_do_not_grow_with_the_batch(precision, storage):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1305_6653_gb300 import FDEBatch, _lib
    counts = []
    for n in (2, 40):
        probs = [fi.random_modes((127, 15)[i % 2], 16, "GBDF3", i) for i in range(n)]
        with FDEBatch(probs) as b:
            b.assemble()
            before = _lib.load().fde_launch_count()
            b.factor(precision, storage=storage)
            counts.append(_lib.load().fde_launch_count() - before)
            xs, stats = b.solve(tol=1e-10, restart=20, maxit=400)
            assert all(st["status"] == 0 for st in stats)
    assert counts[0] == counts[1]
