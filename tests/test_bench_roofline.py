"""The bench's roofline bookkeeping: kernels by what ran, FP32 on the tensor
cores against a sixth of the BF16 rate, shared launches counted once."""

import numpy as np

import bench
from paper_2212_04749_gb300 import tn


def test_peaks_and_launches_by_kernel():
    assert len(bench.FORMS) == 10 and bench.FORMS[tn.TN_FORM_TC_FP32] == "k_step_gemm_tc_bf16x6"
    peaks = {"hbm_gbs": 1000.0, "bf16_tflops_sustained": 600.0, "tf32_tflops": 400.0, "fp32_fma_tflops": 60.0}
    assert bench.compute_peak(tn.TN_FORM_TC_FP32, "fp32", peaks)[0] == 100.0
    assert bench.compute_peak(tn.TN_FORM_TC, "bf16x3", peaks)[0] == 200.0
    assert bench.compute_peak(tn.TN_FORM_TC, "tf32", peaks)[0] == 400.0
    assert bench.compute_peak(tn.TN_FORM_OUTER, "fp32", peaks)[0] == 60.0
    step = {"bytes": 1e6, "flops": 1e9, "runs": 2}
    steps = [dict(step) for _ in range(5)]
    steps[4]["flops"] = 1e12
    forms = np.array([tn.TN_FORM_SMALL] * 3 + [tn.TN_FORM_CHAIN, tn.TN_FORM_TC_FP32])
    roof, frac, dom = bench.roofline_of(steps, np.array([0.0, 0.0, 0.1, 0.2, 40.0]), forms, "fp32", peaks)
    assert dom == tn.TN_FORM_TC_FP32 and roof["bound"] == "tensor" and abs(roof["frac"] - 0.5) < 1e-12
    assert roof["other_families"]["k_small_steps"]["launches"] == 2  # three steps, one launch a batch
    assert roof["other_families"]["k_chain"]["launches"] == 2
