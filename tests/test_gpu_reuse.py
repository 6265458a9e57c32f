"""Problems that come and go: pooled pinned blocks and streams, shared coefficient tables and
merged allocations give the same results for every lifetime, thread and kind of input."""
import threading

import numpy as np
import pytest

import fde_inputs as fi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _solve(prob, precision, **kw):
    from paper_1305_6653_gb300 import FDEProblem
    with FDEProblem.from_inputs(prob, **kw) as p:
        x, st = p.assemble().factor(precision).solve(tol=1e-10)
    assert st["status"] == 0
    return x.cpu().numpy()


def test_results_do_not_depend_on_what_came_before():
    """Four shapes and schemes in turn, twice over, from host and from device arrays, on the
    default and on a side stream, and from four threads at once: the same bits each time."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1305_6653_gb300 import fde_release_cached_memory
    vary = dict(dplus_fn=lambda x: 1.0 + x, dminus_fn=lambda x: 2.0 - x)
    probs = [(fi.manufactured(63, 32, 1.5, "GBDF3", **vary), "fp64"), (fi.manufactured(130, 16, 1.6, "GAM4"), "tf32"),
             (fi.manufactured(40, 64, 1.4, "ETR3", **vary), "fp32"),
             (fi.manufactured_time_varying(63, 16, 1.5, "GBDF5"), "fp64")]
    first = [_solve(p, prec) for p, prec in probs]
    again = [_solve(p, prec, device_inputs=True) for p, prec in probs]
    fde_release_cached_memory()
    side = torch.cuda.Stream()
    other = [_solve(p, prec, stream=side) for p, prec in probs]
    out = [None] * 4

    def work(i):
        s = torch.cuda.Stream()
        out[i] = [_solve(p, prec, stream=s) for p, prec in probs]

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for got in [again, other, *out]:
        for a, b in zip(first, got):
            assert np.array_equal(a, b)


def test_bad_device_inputs_are_refused():
    """Coefficients on the device are checked as the host's are, and a refusal leaves nothing behind."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1305_6653_gb300 import FDEProblem, FdeError
    good = fi.manufactured(50, 16, 1.5, "GBDF3")
    for bad in (-1.0, float("nan"), float("inf")):
        p = fi.manufactured(50, 16, 1.5, "GBDF3")
        p.dplus[17] = bad
        with pytest.raises(FdeError):
            FDEProblem.from_inputs(p, device_inputs=True)
        t = fi.manufactured_time_varying(50, 16, 1.5, "GBDF3")
        t.dminus_t[3, 11] = bad
        for device in (False, True):
            with pytest.raises(FdeError):
                FDEProblem.from_inputs(t, device_inputs=device)
    assert np.isfinite(_solve(good, "fp64", device_inputs=True)).all()
