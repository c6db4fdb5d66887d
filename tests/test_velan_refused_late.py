"""The velocity-analysis loop where the library refuses every step of a later search: the best model found so
far and its history are returned, not lost to the library's error."""
import pytest

from paper_1204_1225_gb300 import kirchhoff as kh
from paper_1204_1225_gb300.velan import VelocityAnalysis


def _loop(objective):
    va = VelocityAnalysis.__new__(VelocityAnalysis)
    va.evaluations = 0
    va.objective = objective
    return va


def _wall(status, after):
    """A slope towards larger v0 whose models are refused after `after` evaluations."""
    calls = []

    def objective(v0, k):
        calls.append((v0, k))
        if len(calls) > after:
            raise kh.KirchhoffError(status, "refused")
        return -1e-3 * v0, -1e-3, 0.0
    return objective, calls


@pytest.mark.parametrize("status", [kh.KH_ERR_UNSUPPORTED, kh.KH_ERR_INVALID_ARG])
@pytest.mark.parametrize("after", [2, 4])
def test_ends_at_the_last_accepted_model(status, after):
    objective, calls = _wall(status, after)
    r = _loop(objective).run(1700.0, 0.5, n_iter=30)
    assert len(r["history"]) == after
    assert (r["v0"], r["k"], r["V"]) == r["history"][-1]
    assert (r["v0"], r["k"]) == calls[after - 1] and r["v0"] > 1700.0
    assert len(calls) - after == 11   # a whole step and ten halvings


def test_other_errors_still_end_the_loop_at_once():
    objective, calls = _wall(kh.KH_ERR_OOM, 3)
    with pytest.raises(kh.KirchhoffError):
        _loop(objective).run(1700.0, 0.5, n_iter=30)
    assert len(calls) == 4


@pytest.mark.parametrize("after", [0, 1])
def test_a_refused_start_or_first_search_raises(after):
    objective, _ = _wall(kh.KH_ERR_UNSUPPORTED, after)
    with pytest.raises(kh.KirchhoffError):
        _loop(objective).run(1700.0, 0.5)
