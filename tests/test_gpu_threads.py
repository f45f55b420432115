"""Solves of different sizes from several threads at once.  A kernel's limit of
dynamic shared memory belongs to the function, not to a launch: a launcher that
sets it to what its own launch needs takes it away from another thread's launch
of a larger size between that thread's setting and its launch, which then fails
with an invalid value."""
import threading

import numpy as np
import pytest

import workloads
from gpu_helpers import write_pinned_tune_cache

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _beside(small, big):
    """Runs small() again and again in another thread while big() runs; big()'s result."""
    stop, errors = threading.Event(), []

    def loop():
        try:
            while not stop.is_set():
                small()
        except Exception as e:   # shown by the assertion below
            errors.append(e)

    t = threading.Thread(target=loop)
    t.start()
    try:
        r = big()
    finally:
        stop.set()
        t.join()
    assert not errors, errors
    return r


def test_fp64_solves_of_two_plans():
    """1000 spots need 60 KB of shared memory, 10 spots 38 KB."""
    from paper_2003_05293_gb300 import Plan
    big, small = (workloads.problem(64, N, 5.0, 0.25, I, seed=N) for N, I in ((1000, 300), (10, 2)))
    with Plan(precision="fp64") as p, Plan(precision="fp64") as q:
        alone = p.solve(big.xyz, 64, big.c, big.iterations, big.seed, state=True)
        r = _beside(lambda: q.solve(small.xyz, 64, small.c, small.iterations, small.seed),
                    lambda: p.solve(big.xyz, 64, big.c, big.iterations, big.seed, state=True))
    assert r["e"] == alone["e"] and np.array_equal(r["theta"], alone["theta"])


def test_serving_beside_new_batches(tmp_path):
    """The serving loop draws masks of P = 1152 (170 KB of shared memory) while the
    caller's thread makes batches of P = 64 (9 KB) on the same plan."""
    from paper_2003_05293_gb300 import Plan
    pbs = [workloads.problem(1152, 16, 5.0, 0.125, 40, seed=s) for s in range(12)]
    small = [workloads.problem(64, 8, 5.0, 0.25, 8, seed=s) for s in range(12)]
    with Plan(precision="fp32", max_batch=16, tune_cache=write_pinned_tune_cache(tmp_path / "t.json", 1, 1, 2)) as p:

        def serve():
            tickets = [p.submit(pb, None) for pb in pbs]
            return [p.wait(t, 60.0) for t in tickets]

        got = _beside(lambda: p.batch(small, None).close(), serve)
    assert all(g["status"] == 0 and 0.0 < g["u"] <= 1.0 for g in got)
