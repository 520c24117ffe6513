"""bench.py asks the plan which kernels a sum takes: stages, launches and the spread variant, on plans made up here."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


class _Points:
    shape = (60000, 30)


class _Plan:
    d, G, P = 30, 256, 1280

    def __init__(self, proj, line):
        self.proj, self.line, self.tuned = proj, line, 0

    def lanes(self, n):
        return n >= self.line

    def autotune(self, x, w):
        self.tuned += 1
        return "moment"

    def set_variant(self, v):
        self.variant = v


class _Problem:
    N, M, P, d, window, n_ft, kernel = 60000, 5000, 1280, 30, 8, 128, "gauss"


@pytest.mark.parametrize("proj,line,stages,launches", [
    ("fp32", 10000, {"project_y"}, 1 + 3 + 2), ("fp32", 1000, set(), 3 + 2), ("fp32", 1 << 30, {"project_x", "project_y"}, 2 + 2 + 2),
    ("fp32_fused", 1000, set(), 3 + 2), ("fp32_fused", 1 << 30, set(), 2 + 2)])
def test_stages_and_launches_by_the_route(proj, line, stages, launches):
    import bench

    ms = {"project_x": 0.005, "project_y": 5.0, "spread_filter": 1.0, "interp": 1.0}  # however short or long they look
    rl = bench.stage_rooflines(_Problem, _Plan(proj, line), ms, {"sm_mhz": 2070.0}, {"bf16_tflops": 1900.0, "hbm_gbs": 6800.0}, "measured", 152)
    assert {k for k in rl if k.startswith("project")} == stages
    assert (rl["spread_filter"]["bound"] == "hbm") == ("project_x" in stages)
    assert (rl["interp"]["bound"] == "hbm") == ("project_y" in stages)
    assert bench.launches_per_step(_Plan(proj, line), _Problem.N, _Problem.M) == launches


def test_launches_of_the_tensor_core_forms():
    import bench

    assert bench.launches_per_step(_Plan("bf16x3", 1000), 60000, 60000) == 9
    assert bench.launches_per_step(_Plan("bf16x3", 1 << 30), 60000, 60000) == 8
    assert bench.launches_per_step(_Plan("tf32", 1 << 30), 4096, 60000) == 7


def test_variant_is_tuned_only_where_there_is_one():
    import bench

    lane, point = _Plan("fp32", 1000), _Plan("fp32", 1 << 30)
    assert bench.tuned_variant(lane, _Points, None) == "slice per lane" and lane.tuned == 0
    assert bench.tuned_variant(point, _Points, None) == "moment" and point.tuned == 1
    assert bench.tuned_variant(point, _Points, None, "tap") == "tap" and point.variant == "tap"
    assert bench.tuned_variant(lane, _Points, None, "tap") == "slice per lane"
