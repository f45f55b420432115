"""The autotuner's choices: what it times, and when it chooses the tensor cores."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("polls", [1, 64])
def test_bounded_wait_test_does_not_reach_the_tuning(polls):
    """Tuning times kernels that do their work, also while the plan's test of the
    bounded waits is on: a tensor-core kernel whose first work item is held back
    takes as long as its waits last (a few microseconds or many times its work),
    and the choice made on it would stay in the plan and its cache file."""
    from paper_2003_05293_gb300 import Plan
    with Plan(precision="fp32") as p:
        ms = p.autotune(1152, 1000, 0.125)
    with Plan(precision="fp32") as p:
        p.test_waits(True, polls)
        held = p.autotune(1152, 1000, 0.125)
        p.test_waits(False, 0)
    assert 0.5 * ms < held < 2.0 * ms
