"""The bench line names the SYRK kernel by the handle's route, not by its rate."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench


def test_slow_slices_are_slices():
    for rate in (0.5 * bench.FP64_PEAK_GFLOPS, 20.0 * bench.FP64_PEAK_GFLOPS, None):
        tensor, kernel, peak, done = bench.syrk_route(5, rate)
        assert tensor and "k_sg_syrk" in kernel and peak == bench.bf16_sustained_tflops() * 1e3
        assert done == (rate * bench.SLICE_PRODUCTS if rate else None)
        assert bench.syrk_route(4, rate) == (False, "k_syrk", bench.FP64_PEAK_GFLOPS, rate)
