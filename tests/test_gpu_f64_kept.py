"""Kept slices of a constant operand in contractions that cut it into different chunks, the second without room for other
slices: both results are right (the second falls back to the CUDA cores before anything is computed).

Tolerance: FP64 sums of 240 real products of entries of order one, a largest result above 20: 240 roundings of 2^-53 of
at most 60 are below 1e-13 of it.
"""
import pytest

from paper_2604_12914_gb300 import binding


@pytest.mark.gpu
@pytest.mark.parametrize("seed", [1, 2])
def test_kept_slices_in_other_chunks(seed):
    first, second = binding.cc_lr_selftest_f64_kept(seed)
    assert first < 1e-13
    assert second < 1e-13
