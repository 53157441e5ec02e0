"""The FP64 passes' fraction of the FP64 peak counts what runs on the FP64 pipe
(the transforms run on the integer pipes): 60 and 25 flops per pixel."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def test_fp64_fraction_counts_the_fp64_pipe():
    r = bench.roofline("fp64", 512, 8, 0.205, 0.330, 1.05, "measured", 0)
    n = 8 * 512 * 512
    for k, flops, ms in (("row", 60, 0.330), ("col", 25, 0.205)):
        p = r["passes"][k]
        assert p["fp64_alu_work_per_launch"] == flops * n
        assert abs(p["frac"] - flops * n / (ms * 1e-3) / 1e12 / 1.05) < 1e-12 and p["frac"] < 1
    assert r["frac"] == r["passes"]["row"]["frac"] and "FP64 pipe" in r["timing"]
