"""Round pupils through the tensor-core kernel with two groups of u warps (short
launches, or more than 128 spots): tiles outside the pupil keep one group busy
with the map's zeros while the pipeline goes on to the other group's tiles.
Every run ends without a wait running out and gives the same numbers, the
oracle's."""
import numpy as np
import pytest

import oracle
import workloads
from gpu_helpers import TOL_EU, write_pinned_tune_cache

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SUBSET_TC, FULL_WS = 1, 2


@pytest.mark.parametrize("P,N,count,strip", [(640, 64, 16, None), (1152, 36, 1, None), (1152, 36, 3, 1), (320, 20, 40, 2),
                                             (512, 130, 24, None), (200, 10, 64, 1)])
def test_runs_end_and_agree(tmp_path, P, N, count, strip):
    from paper_2003_05293_gb300 import Plan
    pbs = [workloads.problem(P, N, 5.0, 0.125, 4, seed=20 + i) for i in range(count)]
    for pb in pbs:
        pb.extra = dict(aperture="round", waist=0.5 * P)
    outs = [torch.empty(pb.M, dtype=torch.float32, device="cuda") for pb in pbs]
    cache = write_pinned_tune_cache(tmp_path / "t.json", SUBSET_TC, 1, FULL_WS, strip=strip)
    with Plan(precision="fp32", max_batch=64, tune_cache=cache) as plan:
        b = plan.batch(pbs, outs)
        seen = set()
        for _ in range(30):
            b.run()
            seen.add(tuple((r["e"], r["u"]) for r in b.results()))   # raises when a wait ran out
        b.close()
    assert len(seen) == 1
    e, u = next(iter(seen))[0]
    ref = oracle.solve(P, pbs[0].xyz, c=pbs[0].c, iterations=4, seed=pbs[0].seed, aperture="round", waist=0.5 * P)
    assert abs(e - ref["e"]) < TOL_EU and abs(u - ref["u"]) < TOL_EU
    edge = outs[0].cpu().numpy().reshape(P, P)[: P // 16, : P // 16]   # a corner outside the pupil
    assert np.all(edge == 0.0)
