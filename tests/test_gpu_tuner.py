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


def test_kernels_of_fp32_products_where_the_tensor_cores_hardly_win(tmp_path):
    """A choice of the tensor cores (products of 16-bit halves) needs more than a
    lead of a few percent over the FP32 kernels: full passes at P = 64, N = 10
    (65 us against 66 for three), a compressed iteration at P = 512, N = 100 (23
    against 24).  Where they win clearly they stay: P = 1152, N = 100 (28
    against 48; full passes 92 against 300)."""
    import json
    from paper_2003_05293_gb300 import Plan
    path = tmp_path / "t.json"
    with Plan(precision="fp32", tune_cache=str(path)) as p:
        for P, N, c in ((64, 10, 0.25), (512, 100, 0.125), (1152, 100, 0.125)):
            p.autotune(P, N, c)
    picks = json.loads(path.read_text())["entries"]
    assert picks["P128_N16_B1_c2"][0] > 3 and picks["P128_N16_B1_c2"][2] > 2
    assert picks["P512_N128_B1_c3"][0] > 3
    assert picks["P1152_N128_B1_c3"][0] == 1 and picks["P1152_N128_B1_c3"][2] == 2


def test_round_pupils_are_tuned_on_round_pupils(tmp_path):
    """A round pupil or a Gaussian beam has a tuning of its own (fewer pixels, dearer
    draws than the square's); entries of cache files written before the pupil was
    in their keys hold for every pupil, as they did."""
    import json
    import workloads
    from gpu_helpers import write_pinned_tune_cache
    from paper_2003_05293_gb300 import Plan
    square, rnd = (workloads.problem(256, 20, 5.0, 0.25, 3, seed=1) for _ in range(2))
    rnd.extra = dict(aperture="round", waist=120.0)
    path = tmp_path / "new.json"
    for first in (square, rnd):   # the second plan finds the first one's file
        with Plan(precision="fp32", tune_cache=str(path)) as p:
            p.batch([first], None).close()
    d = json.loads(path.read_text())
    assert d["format"] == "cswgs-tune-4" and set(d["entries"]) == {"P256_N32_B1_c2", "P256_N32_B1_c2_R_G"}
    path = write_pinned_tune_cache(tmp_path / "old.json", 1, 1, 2)
    with Plan(precision="fp32", tune_cache=path) as p:
        b = p.batch([rnd], None)
        assert b.tile_shape()["threads"] == 1 and b.tile_shape()["full_threads"] == 2
        b.close()
