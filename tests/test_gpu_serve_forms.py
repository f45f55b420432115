"""The forms a served request takes: its compressed iterations on the loop's own
kernel or, when it is much heavier than the loop's first request, on the tensor
cores; without the subset mask, or without the tensor cores' tables, when they
do not fit the loop's memory.  The form shows in the memory that the request
holds (cswgs_serve_stats), and the heavy ones keep the precision of the FP32
phasors that they would have run on."""
import time

import numpy as np
import pytest

import workloads
from gpu_helpers import TOL_EU, write_pinned_tune_cache

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DIRECT, FULL_WS = 128, 2


def _plan(tmp_path, cap):
    from paper_2003_05293_gb300 import Plan
    return Plan(precision="fp32", max_batch=16, mem_cap_bytes=cap,
                tune_cache=write_pinned_tune_cache(tmp_path / "t.json", DIRECT, 8, FULL_WS))


def _held(p, pb):
    """Memory that the loop holds for this request alone, and its result."""
    long = workloads.problem(pb.P, pb.N, 5.0, pb.c, 20000, seed=1)   # runs until it is cancelled
    assert p.serve_stats()["bytes_in_use"] == 0
    t, end = p.submit(long, None), time.time() + 20.0
    held = 0
    while held == 0 and time.time() < end:
        held = p.serve_stats()["bytes_in_use"]
    p.cancel(t)
    p.wait(t)
    return held, p.wait(p.submit(pb, None))


def test_forms_by_memory(tmp_path):
    light = workloads.problem(256, 10, 5.0, 0.125, 3, seed=1)
    heavy = workloads.problem(512, 64, 5.0, 0.125, 3, seed=2)    # c N = 8 a spot block
    mask = 512 * 512 // 8                                        # a bit per pixel
    cap, held = 1 << 30, []
    for _ in range(3):
        with _plan(tmp_path, cap) as p:
            p.wait(p.submit(light, None))
            h, r = _held(p, heavy)
            ref = p.solve(heavy.xyz, heavy.P, heavy.c, heavy.iterations, heavy.seed)
        assert abs(r["e"] - ref["e"]) < TOL_EU and abs(r["u"] - ref["u"]) < TOL_EU
        held.append(h)
        cap = h - 256    # the next loop has no room for this form
    tables, bare, lean = held
    assert tables - bare == mask        # the tensor cores for compressed iterations, then the loop's own kernel
    assert 0 < lean < bare - 4 * 64 * 512   # no factor tables at all


def test_a_light_request_stays_on_the_loops_kernel(tmp_path):
    """c N = 4 a spot block is the line: N = 32 at c = 1/8 holds no mask, N = 33 does."""
    per_spot, held = None, {}
    with _plan(tmp_path, 1 << 30) as p:
        p.wait(p.submit(workloads.problem(256, 10, 5.0, 0.125, 3, seed=1), None))
        for N in (31, 32, 33, 34):
            held[N] = _held(p, workloads.problem(256, N, 5.0, 0.125, 3, seed=N))[0]
    per_spot = held[34] - held[33]
    assert held[32] - held[31] <= per_spot + 2048
    assert held[33] - held[32] >= 256 * 256 // 8


def test_heavy_requests_keep_their_precision(tmp_path):
    """u after 40 iterations against the FP64 solver: served on the tensor cores
    within twice (a handful of holograms' scatter) of the same holograms on FP32
    phasors.  With a strip dot whose recurrence is off by the hardware's sine it
    is 5 times as far off."""
    from paper_2003_05293_gb300 import Plan
    pbs = [workloads.problem(384, 150, 10.0, 0.25, 40, seed=50 + s) for s in range(8)]
    with Plan(precision="fp64") as f, _plan(tmp_path, 1 << 30) as p:
        exact = np.array([f.solve(pb.xyz, pb.P, pb.c, pb.iterations, pb.seed)["u"] for pb in pbs])
        direct = np.array([p.solve(pb.xyz, pb.P, pb.c, pb.iterations, pb.seed)["u"] for pb in pbs])
        p.wait(p.submit(workloads.problem(384, 10, 5.0, 0.25, 3, seed=1), None))
        served = np.array([p.wait(t)["u"] for t in [p.submit(pb, None) for pb in pbs]])

    def rms(d):
        return float(np.sqrt(np.mean(d * d)))

    assert rms(served - exact) < 2.0 * rms(direct - exact)
