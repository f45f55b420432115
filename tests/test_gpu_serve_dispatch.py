"""The serving loop's choice of the compressed kernel per request: a loop whose
shape was tuned for a request of few spots runs the heavier requests that
follow on the tensor cores, and a request whose subset mask does not fit the
loop's memory on the shape's own kernel; results as of solo solves."""
import numpy as np
import pytest

import workloads
from gpu_helpers import TOL_EU, write_pinned_tune_cache

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DIRECT, FULL_WS = 128, 2


def _plan(tmp_path, cap):
    from paper_2003_05293_gb300 import Plan
    return Plan(precision="fp32", max_batch=16, mem_cap_bytes=cap, max_N=1024,
                tune_cache=write_pinned_tune_cache(tmp_path / "t.json", DIRECT, 8, FULL_WS))


@pytest.mark.parametrize("cap", [1 << 30, 0])
def test_heavy_requests_after_a_light_one(tmp_path, cap):
    sizes = [(256, 10, 0.125), (256, 100, 0.25), (512, 1000, 0.125), (200, 130, 0.0625), (256, 33, 0.125),
             (256, 32, 0.125)]
    pbs = [workloads.problem(P, N, 5.0, c, 5, seed=300 + i) for i, (P, N, c) in enumerate(sizes)]
    with _plan(tmp_path, cap or (1 << 30)) as p:
        outs = [torch.empty(pb.M, dtype=torch.float32, device="cuda") for pb in pbs]
        tickets = [p.submit(pb, o) for pb, o in zip(pbs, outs)]
        got = [p.wait(t) for t in tickets]
        for pb, g in zip(pbs, got):
            r = p.solve(pb.xyz, pb.P, pb.c, pb.iterations, pb.seed)
            assert abs(g["e"] - r["e"]) < TOL_EU and abs(g["u"] - r["u"]) < TOL_EU


def test_no_room_for_the_mask(tmp_path):
    """A loop with room for the request but not for its mask still takes it."""
    small = workloads.problem(256, 10, 5.0, 0.125, 3, seed=1)
    big = workloads.problem(512, 64, 5.0, 0.125, 3, seed=2)
    with _plan(tmp_path, 1 << 30) as p:
        p.wait(p.submit(small, None))
        before = p.serve_stats()["bytes_in_use"]
        t = p.submit(big, None)
        p.wait(t)
        assert before == 0
        ref = p.solve(big.xyz, big.P, big.c, big.iterations, big.seed)
    lo, hi = 1 << 20, 1 << 26   # the smallest cap that takes the request
    def taken(cap):
        (tmp_path / "q").mkdir(exist_ok=True)
        with _plan(tmp_path / "q", cap) as p:
            try:
                p.wait(p.submit(small, None))
                r = p.wait(p.submit(big, None))
            except Exception:
                return None
            return r
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        if taken(mid) is not None:
            hi = mid
        else:
            lo = mid
    r = taken(hi)
    assert abs(r["e"] - ref["e"]) < TOL_EU and abs(r["u"] - ref["u"]) < TOL_EU


def test_no_room_for_the_tables(tmp_path):
    """A loop whose shape runs everything on the tensor cores takes a request
    whose factor tables do not fit its memory on the CUDA-core kernels, beside
    one that fits, and refuses one that fits neither way."""
    from paper_2003_05293_gb300 import CswgsError, Plan
    cache = write_pinned_tune_cache(tmp_path / "t.json", 1, 1, FULL_WS)
    fits = workloads.problem(64, 8, 2.0, 0.25, 4, seed=5)
    lean = workloads.problem(256, 8, 2.0, 0.25, 4, seed=6)     # 384 KiB without tables, 600 KiB with them
    never = workloads.problem(1024, 8, 2.0, 0.25, 4, seed=7)   # its phase map alone is 4 MiB
    with Plan(precision="fp32", max_batch=8, mem_cap_bytes=500 << 10, tune_cache=cache) as p:
        for pb in (fits, lean, fits):
            g = p.wait(p.submit(pb, None), 60.0)
            r = p.solve(pb.xyz, pb.P, pb.c, pb.iterations, pb.seed)
            assert abs(g["e"] - r["e"]) < TOL_EU and abs(g["u"] - r["u"]) < TOL_EU
        with pytest.raises(CswgsError):
            p.submit(never, None)
