"""The benchmark line's roofline: a launch of the FP64 path runs on the tensor cores, at several times the rate of the FP64
units, and so has no share of theirs."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

DERIVED = {"fp32": 80.5, "sms": 152, "sm_max_ghz": 2.07}
CUBLAS = {"fp32": 69.7, "fp64": 1.1}


@pytest.mark.parametrize("path,tflops,frac", [("fp32", 38.94, 0.4837), ("fp64", 6.5, None)])
def test_share_of_the_peak(path, tflops, frac):
    r = bench.alu_roofline(path, "gemm_M=UK", tflops * 1e10, 10.0, DERIVED, CUBLAS, None)
    assert r["achieved"] == tflops and r["frac"] == frac and (r["peak"] is None) == (frac is None)
    assert r["frac_of_cublas_gemm"] == round(tflops / CUBLAS[path], 4)


def test_no_peak_of_the_fp64_units():
    class Torch:
        class cuda:
            @staticmethod
            def get_device_properties(k):
                return type("P", (), {"multi_processor_count": 152})

    assert "fp64" not in bench.derived_alu_peaks(Torch, 2070.0)
