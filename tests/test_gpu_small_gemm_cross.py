"""Products of a few rows or columns in complex128 on the CUDA cores against another kernel, the 3xTF32 tensor-core GEMM of the same
operands: complex64 and complex128 share their kernel there, so comparing those two with each other cannot show what both
get wrong (an edge tile, a K tail, a split).

The tolerance is the one of the tensor-core GEMM self-test in mode 2 (1e-8 K + 2e-6 of the largest entry).
"""
import pytest

from paper_2604_12914_gb300 import binding


@pytest.mark.gpu
@pytest.mark.parametrize("M,N", [(1, 300), (257, 1), (256, 2), (3, 65), (64, 4), (65, 5), (15, 16), (17, 17), (40, 10)])
@pytest.mark.parametrize("K", [1, 15, 17, 64, 130, 1000])
def test_small_products_against_tensor_cores(M, N, K):
    tc, _ = binding.cc_lr_selftest_gemm(M, N, K, 2, seed=M + N + K)
    assert 0 <= tc < 1e-8 * K + 2e-6
