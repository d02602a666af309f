"""The bench's tensor peak names the clock it was measured at: fractions of a power-limited rate are not the pipe's."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

STATS = {
    "flops_stage": [10.0, 1.0, 40.0, 20.0, 8.0, 2.0], "flops_fp64": 81.0, "flops_term2": 6.0,
    "flops_term1_tc": 30.0, "flops_z_tc": 20.0, "flops_t_tc": 10.0, "tensor_flops": 1e4,
    "tensor_flops_stage": [1e3, 2e3, 3e3, 2.5e3, 1.5e3],
}


def test_peak_source_names_the_clock(monkeypatch):
    gemm = {"ms_per_build": 2.0, "launches_per_build": 4.0, "stage_pairs_per_build": 1000.0}
    r = {"stats": STATS, "stage_ms": {}, "gemm": gemm}
    peaks = {"bf16_tflops_sustained": 1700.0, "clocks_under_load": {"sm_mhz_median": 1485.0}}
    monkeypatch.setattr(bench, "peaks", lambda: (peaks, "measured"))
    assert bench.roofline("mixed", r)["peak_source"].endswith("measured, at a median SM clock of 1485 MHz")
    monkeypatch.setattr(bench, "peaks", lambda: ({"bf16_tflops_sustained": 1700.0}, "fallback"))
    assert bench.roofline("mixed", r)["peak_source"].endswith("fallback")
