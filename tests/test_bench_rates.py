"""bench.py's memory rates for launches of several steps: what a launch moves, not what its steps would
have moved one by one."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_steps_per_launch():
    assert bench.steps_per_launch(600, 100, "f32") == 6
    assert bench.steps_per_launch(100, 100, "bf16") == 1
    assert bench.steps_per_launch(100, 0, "f32", "aa") == 1       # not counted
    # FP16: a step and its scales' update; two steps, the update and the launch that mends
    assert bench.steps_per_launch(100, 200, "f16") == 1
    assert bench.steps_per_launch(100, 150, "f16") == 2
    assert bench.steps_per_launch(101, 2 + 150, "f16") == pytest.approx(101 / 51)


def test_fused_rates_count_a_launch_once(monkeypatch):
    monkeypatch.setattr(bench, "_peaks", lambda: (6000.0, "measured"))
    sites, sec = 4096 * 4096, 1.0
    # D2Q5 FP32, indexed: 41 B a site; 12000 steps a second in launches of 6
    one = bench.hbm_use(5, "f32", True, sites, 12000, 1.0, sec)
    six = bench.hbm_use(5, "f32", True, sites, 12000, 6.0, sec)
    assert one["achieved_gbs"] == one["one_step_equivalent_gbs"] == six["one_step_equivalent_gbs"]
    assert six["achieved_gbs"] == pytest.approx(one["achieved_gbs"] / 6, rel=1e-4)
    assert six["achieved_gbs"] == pytest.approx(41 * sites * 2000 / 1e9, rel=1e-4)
    assert six["frac_of_measured_hbm"] == pytest.approx(six["achieved_gbs"] / 6000, rel=1e-3)


def test_traffic_names_a_kernel_that_exists():
    for (kernel, _), (_, stamp, profile) in bench.NCU_TRAFFIC.items():
        assert bench.source_hash(kernel) is not None
        assert len(stamp) == 12 and os.path.exists(os.path.join(ROOT, profile))
