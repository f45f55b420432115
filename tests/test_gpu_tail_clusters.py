"""Tails of tensor-core launches by clusters of 8, 4, 2 and 1 blocks per
hologram: a launch takes as many as leave every hologram's cluster on SMs of
its own, from 2048 partials a hologram.  Strips are pinned to one tile (50 work
items of 44 to 52 spots), so 12, 20, 40 and 80 holograms take the four sizes.
Each hologram's numbers are those of a solve of its own (a cluster of 8), which
sums the same partials in another order."""
import numpy as np
import pytest

import oracle
import workloads
from gpu_helpers import TOL_EU, write_pinned_tune_cache

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("count", [12, 20, 40, 80])
def test_batch_equals_solves(tmp_path, count):
    from paper_2003_05293_gb300 import Plan
    cache = write_pinned_tune_cache(tmp_path / "t.json", 1, 1, 2, batch_pow2=range(0, 8), strip=1)
    pbs = [workloads.problem(640, 44 + i % 9, 5.0, 0.25, 2, seed=300 + i) for i in range(count)]
    with Plan(precision="fp32", max_batch=128, tune_cache=cache) as p:
        b = p.batch(pbs, None)
        b.run()
        got = b.results()
        b.close()
        for i in range(0, count, 5):
            r = p.solve(pbs[i].xyz, 640, 0.25, 2, pbs[i].seed, state=True)
            # sums of some 50 partials in FP32 with compensation: 1e-7 of each V_n, twice squared
            assert abs(got[i]["e"] - r["e"]) < 2e-6 and abs(got[i]["u"] - r["u"]) < 2e-5
    ref = oracle.solve(640, pbs[0].xyz, c=0.25, iterations=2, seed=pbs[0].seed)
    assert abs(got[0]["e"] - ref["e"]) < TOL_EU and abs(got[0]["u"] - ref["u"]) < TOL_EU
