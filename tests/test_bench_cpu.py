"""The benchmark's derived figures that need no GPU."""
import pytest

import bench


def test_fp64_roofline_names_the_kernels_and_counts_what_they_execute():
    kw = dict(kernel_ms=2.0, peak=1.0, peak_source="measured")
    near = bench.fp64_roofline([(81e9, 1)], **kw)
    assert "apply_f64_sym_kernel" in near["kernel"] and "apply_f64_kernel" not in near["kernel"]
    assert near["achieved"] == pytest.approx(19.5e9 / 2e-3 / 1e12) and near["algorithmic_tflops"] == pytest.approx(40.5)
    wide = bench.fp64_roofline([(1e9, 2)], **kw)
    assert wide["kernel"] == "apply_f64_kernel" and wide["achieved"] == wide["algorithmic_tflops"] == pytest.approx(0.5)
    both = bench.fp64_roofline([(1e9, 3), (81e9, 1)], **kw)
    assert "apply_f64_kernel" in both["kernel"] and "apply_f64_sym_kernel" in both["kernel"]
    assert both["achieved"] == pytest.approx(near["achieved"] + wide["achieved"]) and both["frac"] == both["achieved"]
