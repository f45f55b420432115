"""The double-precision solver at the sizes where its work is split
differently, against the oracle: more spots than a block has threads, grids of
more than one list segment (1024 columns), sparse and empty rows, several rows
per block, one pixel per iteration."""
import math

import numpy as np
import pytest

import oracle
import workloads
from gpu_helpers import TOL_FP64_EU, TOL_FP64_PHASE, rms_wrapped

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def fp64():
    from paper_2003_05293_gb300 import Plan
    p = Plan(precision="fp64")
    yield p
    p.close()


@pytest.mark.parametrize("P,N,c", [(2, 1, 0.25), (32, 513, 0.5), (34, 600, 1.0), (64, 200, 1.0 / 4096), (96, 7, 0.01),
                                   (1026, 3, 0.02), (1250, 2, 0.3), (64, 3100, 0.25)])
def test_iterations_and_metrics(fp64, P, N, c):
    if N > 1024:
        from paper_2003_05293_gb300 import Plan
        fp64 = Plan(precision="fp64", max_N=4096)
    pb = workloads.problem(P, N, 5.0, c, 3, seed=60 + N)
    rng = np.random.default_rng(N)
    w0, th0 = np.exp(rng.normal(0.0, 0.3, N)), rng.uniform(-np.pi, np.pi, N)
    amp = rng.uniform(0.5, 1.5, N)
    # one compressed iteration, then one full one and the metrics
    for I, full, fin in ((1, 0, False), (1, 1, True)):
        r = fp64.solve(pb.xyz, P, c, I, pb.seed, amp=amp, init_w=w0, init_theta=th0, first_iteration=2,
                       full_iterations=full, final_pass=fin, state=True)
        ref = oracle.solve(P, pb.xyz, amp, c=c, iterations=I, seed=pb.seed, theta_in=th0, w_in=w0, first_j=2,
                           full_iterations=full, final_pass=fin)
        assert rms_wrapped(r["theta"], ref["theta"]) < TOL_FP64_PHASE
        assert math.sqrt(np.mean((r["w"] / ref["w"] - 1) ** 2)) < TOL_FP64_PHASE
        if fin:
            assert abs(r["e"] - ref["e"]) < TOL_FP64_EU and abs(r["u"] - ref["u"]) < TOL_FP64_EU
