"""Outputs of the tensor-core kernel against recorded ones (golden/tc_outputs.npz):
a whole solve, a final pass of 300 spots, and one with whole-row strips, at P =
1152 on pinned launch shapes.  What a caller gets for the same inputs stays
within FP32 rounding of what it was; a change of the arithmetic, also one
towards exact values, shows here.  The bounds: an FP32 sum's rounding is 6e-8 of
a value, and the sums behind an output are a few such roundings deep."""
import os

import numpy as np
import pytest

import workloads
from gpu_helpers import rms_wrapped, wrap, write_pinned_tune_cache

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SUBSET_TC, FULL_WS = 1, 2
TOL_E = 1e-6          # relative
TOL_I_SPREAD = 1e-6   # rms over spots of I_n over its recorded value, the mean apart
TOL_THETA = 1e-5      # rad rms after 30 iterations
TOL_MAP_RMS, TOL_MAP_MAX = 1e-6, 2e-5   # rad; a pixel whose |S| is 1 / 100 of the mean has 100 times the rounding


@pytest.fixture(scope="module")
def golden(golden_dir):
    return np.load(os.path.join(golden_dir, "tc_outputs.npz"))


def _plan(tmp_path_factory, strip=None):
    from paper_2003_05293_gb300 import Plan
    path = tmp_path_factory.mktemp("out") / "t.json"
    return Plan(precision="fp32", tune_cache=write_pinned_tune_cache(path, SUBSET_TC, 1, FULL_WS, strip=strip))


def _state(N, seed):
    rng = np.random.default_rng(seed)
    return np.exp(rng.normal(0.0, 0.3, N)), rng.uniform(-np.pi, np.pi, N)


@pytest.fixture(scope="module")
def solve(tmp_path_factory):
    pb = workloads.problem(1152, 100, 10.0, 0.125, 30, seed=41)
    with _plan(tmp_path_factory) as p:
        return p.solve(pb.xyz, pb.P, pb.c, 30, pb.seed, state=True)


@pytest.fixture(scope="module")
def final(tmp_path_factory):
    pb = workloads.problem(1152, 300, 10.0, 1.0, 0, seed=42)
    w, th = _state(300, 6)
    out = torch.empty(pb.M, device="cuda")
    with _plan(tmp_path_factory) as p:
        r = p.solve(pb.xyz, pb.P, 1.0, 0, pb.seed, init_w=w, init_theta=th, out=out, state=True)
    r["map"] = out.cpu().numpy()[np.random.default_rng(7).choice(pb.M, 8192, replace=False)]
    return r


def test_efficiency(golden, solve, final):
    assert abs(solve["e"] / golden["solve_eu"][0] - 1) < TOL_E
    assert abs(final["e"] / golden["final_eu"][0] - 1) < TOL_E


def test_intensities(golden, final):
    assert np.std(final["I"] / golden["final_I"]) < TOL_I_SPREAD


def test_spot_phases(golden, solve):
    assert rms_wrapped(solve["theta"], golden["solve_theta"]) < TOL_THETA


def test_phase_map(golden, final):
    d = wrap(final["map"].astype(np.float64) - golden["final_map"])
    assert np.sqrt(np.mean(d * d)) < TOL_MAP_RMS and np.abs(d).max() < TOL_MAP_MAX


def test_whole_row_strips(golden, tmp_path_factory):
    """Strips pinned to a row block's 18 tiles: the accumulation over them drops
    1.1e-5 of e, over half as many 4e-6."""
    pb = workloads.problem(1152, 100, 10.0, 1.0, 0, seed=43)
    w, th = _state(100, 8)
    with _plan(tmp_path_factory, strip=18) as p:
        r = p.solve(pb.xyz, pb.P, 1.0, 0, pb.seed, init_w=w, init_theta=th, state=True)
    assert abs(r["e"] / golden["rows_eu"][0] - 1) < TOL_E
