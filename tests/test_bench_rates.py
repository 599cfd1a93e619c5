"""The benchmark's per-kind figures: kinds that do all of Algorithm 2's multiply-adds have a
fraction of the pipe's rate, kinds that skip most of them only the algorithm's count per second."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def timing(ms, work):
    return {"ms": ms, "launches": 2, "work": work}


STEP = {"stagej_fp32": timing(2.0, 10 ** 10), "stage0_fp64": timing(1.0, 10 ** 8),
        "leaf_fp32": timing(4.0, 6 * 10 ** 10), "leaf_fp64": timing(3.0, 2 * 10 ** 9),
        "leaf_pair": timing(0.5, 10 ** 9), "leaf_midrad": timing(1.0, 10 ** 9),
        "split": timing(1.0, 5 * 10 ** 9), "compact": {"ms": 0.0, "launches": 0, "work": 0}}


def test_kinds_that_skip_operations_have_no_fraction():
    out = bench.roofline_by_kind([STEP, STEP], 40.0, 0.6, 7000.0)
    assert set(out) == set(STEP) - {"compact"}
    for name in ("leaf_fp32", "leaf_fp64", "leaf_pair"):
        assert "frac" not in out[name] and "achieved" not in out[name]
        w, ms = STEP[name]["work"], STEP[name]["ms"]
        assert abs(out[name]["algorithmic_madds_per_s"] / (w / (ms * 1e-3)) - 1) < 1e-12
    for name, peak in (("stagej_fp32", 40.0), ("stage0_fp64", 0.6), ("leaf_midrad", 40.0)):
        want = 4 * STEP[name]["work"] / (STEP[name]["ms"] * 1e-3) / 1e12 / peak
        assert abs(out[name]["frac"] / want - 1) < 1e-12
        assert out[name]["madds_per_step"] == STEP[name]["work"]
    assert abs(out["split"]["frac"] / (5 * 10 ** 9 / 1e-3 / 1e9 / 7000.0) - 1) < 1e-12
    assert out["split"]["bytes_per_step"] == STEP["split"]["work"]
    assert abs(sum(v["time_share"] for v in out.values()) - 1) < 1e-12


def test_the_top_kernel_has_no_fraction_either_where_it_skips():
    top = bench.roofline([STEP, STEP], 40.0, 0.6)
    assert top["kernel"] == "leaf_fp32" and "frac" not in top and top["traffic"] > 0
    assert top["launches"] == 4 and top["avg_launch_ms"] == 2.0
    assert abs(sum(top["time_share"].values()) - 1) < 1e-3
    top = bench.roofline([{"stagej_fp32": timing(2.0, 10 ** 10), "leaf_fp32": timing(1.0, 1)}], 40.0, 0.6)
    assert top["kernel"] == "stagej_fp32" and top["frac"] > 0 and top["traffic"] is None
