"""The FP64 tensor-core GEMM (exact 8-bit slices) against extended-precision sums on the host, at the
edges of its tiles (128 rows; 16, 32 or 64 complex columns), of its K chunks (16 complex) and of its
operand layouts, over scales from 2^-300 to 2^300, and with a NaN.

Bound (the library divides by it, so the limit here is 1): the result is rounded a few times in FP64
(8 u covers the rounding of the sum, of alpha and of the addition to C), and every product of two real
entries loses at most 9.2 * 2^-64 of (largest entry of the row) x (largest entry of the column), 2 K of
them per sum: less than K 2^-59; the float that holds orders 5-7 (below 2^-40) is rounded once per
chunk of 32: at most K^2 2^-67.
"""
import pytest

from paper_2604_12914_gb300 import binding


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (5, 3, 16), (127, 16, 17), (128, 17, 15), (129, 32, 33), (130, 33, 64),
                                   (200, 64, 90), (257, 65, 130), (40, 130, 700), (300, 10, 2100), (7, 7, 5000)])
@pytest.mark.parametrize("layout", [0, 1, 2, 3, 4, 15])
def test_f64_gemm_within_bound(M, N, K, layout):
    err, nans = binding.cc_lr_selftest_f64gemm(M, N, K, layout, spread=20.0, seed=M + 7 * N + K)
    assert err <= 1.0, err
    assert nans == 0


@pytest.mark.gpu
@pytest.mark.parametrize("layout", [0, 3])
def test_f64_gemm_wide_scales_and_nan(layout):
    err, nans = binding.cc_lr_selftest_f64gemm(150, 70, 40, layout, spread=300.0, seed=3)
    assert err <= 1.0, err
    assert nans == 0
    err, nans = binding.cc_lr_selftest_f64gemm(150, 70, 40, layout | 16, seed=4)
    assert err <= 1.0, err
    assert nans == 0
