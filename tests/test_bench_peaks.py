"""The tensor peaks that bench.py's rooflines are fractions of, from the measured rates of what the kernels
issue: six bf16 products per fp32 product, four TF32 ones in the QR's block updates, one bf16 product in
Muon."""
import bench

PEAKS = {"hbm_gbs": 6778.7, "bf16_tflops": 1907.4, "bf16_tflops_sustained": 1728.0}
ABOVE_THE_RIDGE = {"ms": 100.0, "launches": 10, "flops": 20e12, "bytes": 50e9}


def test_tensor_peak_of_each_family():
    peak = lambda family, **kw: bench.roofline(family, ABOVE_THE_RIDGE, PEAKS, "measured", **kw)["peak"]  # noqa: E731
    assert abs(peak("gemm_tc") - 1728.0 / 6) < 1e-9
    assert abs(peak("qr_update") - bench.TF32_TFLOPS["sustained"] / 4) < 1e-9
    assert peak("gemm_tc", products=1) == 1728.0
