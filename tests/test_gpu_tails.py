"""The tails of the tensor-core launches (weighted update, metrics) and the
amplitude range of their operands, at the sizes where the work's split
changes: spots dealt out in fours to 1 to 8 blocks per hologram and to 1 to
16 warps per four spots (N below, at and past multiples of 4, 32 and 128; few
and many work items; one hologram and batches of 3, 20 and 80), against the
oracle, teacher-forced."""
import math

import numpy as np
import pytest

import oracle
import workloads
from gpu_helpers import TOL_EU, TOL_PHASE_RMS, rms_wrapped, write_pinned_tune_cache

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SUBSET_TC, FULL_WS = 1, 2


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    from paper_2003_05293_gb300 import Plan
    path = tmp_path_factory.mktemp("tails") / "t.json"
    p = Plan(precision="fp32", max_batch=128, tune_cache=write_pinned_tune_cache(path, SUBSET_TC, 1, FULL_WS,
                                                                                 batch_pow2=range(0, 8)))
    yield p
    p.close()


def _start(N, seed):
    rng = np.random.default_rng(seed)
    return np.exp(rng.normal(0.0, 0.3, N)), rng.uniform(-np.pi, np.pi, N)


@pytest.mark.parametrize("P,N", [(64, 1), (64, 3), (128, 4), (130, 5), (256, 33), (256, 127), (300, 129), (640, 31),
                                 (200, 1000)])
@pytest.mark.parametrize("full", [0, 1])
def test_update_and_metrics(plan, P, N, full):
    pb = workloads.problem(P, N, 5.0, 0.25, 1, seed=40 + N)
    w0, th0 = _start(N, N)
    r = plan.solve(pb.xyz, P, pb.c, 1, pb.seed, init_w=w0, init_theta=th0, first_iteration=3, full_iterations=full,
                   final_pass=True, state=True)
    ref = oracle.solve(P, pb.xyz, c=pb.c, iterations=1, seed=pb.seed, theta_in=th0, w_in=w0, first_j=3,
                       full_iterations=full)
    assert rms_wrapped(r["theta"], ref["theta"]) < TOL_PHASE_RMS
    assert math.sqrt(np.mean((r["w"] / ref["w"] - 1) ** 2)) < TOL_PHASE_RMS
    assert abs(r["e"] - ref["e"]) < TOL_EU and abs(r["u"] - ref["u"]) < TOL_EU
    assert abs(float(np.sum(r["I"])) - r["e"]) < 1e-12 * N


@pytest.mark.parametrize("count", [3, 12, 20, 80])
def test_batch_tails_and_masks(plan, count):
    """Batches that take clusters of 8, 4 and 1 blocks (12: 8 again), and subset masks drawn
    in global memory or in the shared memory of 8, 4 and 1 blocks: each hologram
    of uneven size against the oracle.  (N = 2 would hang on pixels where S
    vanishes, whose phase is arbitrary to any rounding.)"""
    rng = np.random.default_rng(count)
    pbs = []
    for i in range(count):
        pb = workloads.problem(int(rng.choice([64, 98, 160, 258])), int(rng.integers(5, 40)), 5.0, 0.25, 4,
                               seed=900 + i)
        if i % 3 == 1:
            pb.extra = dict(aperture="round", waist=0.6 * pb.P, subset_mode="windows" if i % 2 else "fresh")
        pbs.append(pb)
    b = plan.batch(pbs, None)
    b.run()
    got = b.results()
    b.close()
    for pb, g in zip(pbs, got):
        ex = getattr(pb, "extra", None) or {}
        ref = oracle.solve(pb.P, pb.xyz, c=pb.c, iterations=pb.iterations, seed=pb.seed, **(
            dict(aperture=ex["aperture"], waist=ex["waist"], subset_mode=ex["subset_mode"]) if ex else {}))
        assert abs(g["e"] - ref["e"]) < TOL_EU and abs(g["u"] - ref["u"]) < TOL_EU


@pytest.mark.parametrize("scale", [1e-25, 1e-12, 1.0, 1e18])
def test_amplitude_scale(plan, scale):
    """u = S / |S| and the phase map do not depend on the amplitudes' scale, also
    where |S|^2 leaves FP32's normal range; a weak spot among strong ones keeps
    its phase."""
    P, N = 192, 20
    pb = workloads.problem(P, N, 5.0, 0.25, 3, seed=77)
    amp = np.linspace(0.5, 1.5, N) * scale
    amp[3] *= 1e-3
    out = torch.empty(pb.M, dtype=torch.float32, device="cuda")
    r = plan.solve(pb.xyz, P, pb.c, 3, pb.seed, amp=amp, out=out, state=True)
    ref = oracle.solve(P, pb.xyz, amp / scale, c=pb.c, iterations=3, seed=pb.seed)
    assert rms_wrapped(r["theta"], ref["theta"]) < TOL_PHASE_RMS
    assert rms_wrapped(out.cpu().numpy(), ref["phase"]) < TOL_PHASE_RMS
    assert abs(r["e"] - ref["e"]) < TOL_EU and abs(r["u"] - ref["u"]) < TOL_EU
