"""The bench's roofline of the K1 contraction: both forms run on the FP16 tensor cores, with
3 (hi + lo) or 11 (slices and their guard) products per algorithmic flop, and are
compared with that peak."""
import numpy as np
import pytest

import bench


@pytest.mark.parametrize("tc,products", [(1, 3.0), (0, 11.0)])
def test_compared_with_the_tensor_peak(tc, products):
    peaks = {"bf16_tflops_sustained": 1700.0, "hbm_gbs": 6800.0}
    ms, fl, by = np.array([1.0, 2.0]), np.array([1e11, 2e11]), np.array([1e6, 1e6])
    r = bench.roofline({"ms": 3.0, "flops": 3e11, "launches": 2}, ms, fl, by, peaks, "measured", tc, 10.0)
    assert r["bound"] == "tensor" and r["peak"] == 1700.0
    assert r["achieved"] == pytest.approx(100.0)
    assert r["mma_pipe_frac"] == pytest.approx(products * 100.0 / 1700.0)
    assert r["attainable_frac"] == pytest.approx(products * 100.0 / 1700.0)
    assert r["mma_pipe_frac"] <= 1.0
