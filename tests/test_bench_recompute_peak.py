"""The recompute peak of the bench line is that of the path that runs: the residual
as 17 FP16 plane products and the correction as three TF32 products, both on the
tensor cores (no GPU)."""
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_recompute_peak_with_the_correction_on_the_tensor_cores():
    import bench
    from paper_1901_01047_gb300 import inputs
    peaks = {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0}
    r = bench.roofline("recompute", 1000.0, 10, {"recompute": (None, 2.0e12)}, peaks, "measured",
                       inputs.WORKLOADS["batched256"], correction="tf32x3")
    # 4 n^3 flop: 17 products of 2 n^3 at the 16-bit rate, 3 of 2 n^3 at the TF32 rate
    assert r["peak"] == pytest.approx(4.0 / (2.0 * 17 / 1700.0 + 2.0 * 3 / (1700.0 * 1.1 / 2.25)))
    assert r["frac"] == pytest.approx(2.0 / r["peak"]) and "TF32" in r["peak_kind"]


def test_bench_line_uses_it():
    with open(os.path.join(ROOT, "paper_1901_01047_gb300", "csrc", "k_aux.cu")) as f:
        assert "launch_correct_tc(cfg, st);" in f.read()  # the correction of the default recompute
    with open(os.path.join(ROOT, "bench.py")) as f:
        calls = re.findall(r'roof\w* = roofline\((?:dominant|"recompute"),[^)]*\)', f.read())
    assert len(calls) == 2 and all('correction="tf32x3"' in c for c in calls)
