"""Products of a few rows or columns on the CUDA cores (one output per thread, 16 x 16, 64 x 4 and 256 x 1
tiles, K split over blocks), complex64 against complex128, at the edges of the tiles and of the K blocks.

The tolerance is the one of the tensor-core GEMM self-test for the FP32 CUDA cores (2e-5 of the largest
entry; FP32 sums of at most 64 products per split).
"""
import pytest

from paper_2604_12914_gb300 import binding


@pytest.mark.gpu
@pytest.mark.parametrize("M,N", [(1, 1), (1, 300), (257, 1), (256, 2), (3, 65), (64, 4), (65, 5), (15, 16), (17, 17), (40, 10)])
@pytest.mark.parametrize("K", [1, 15, 17, 64, 130, 1000])
def test_small_products(M, N, K):
    tc, fp32 = binding.cc_lr_selftest_gemm(M, N, K, 2, seed=M + N + K)
    assert 0 <= fp32 < 2e-5


@pytest.mark.gpu
@pytest.mark.parametrize("M,N", [(700, 650), (13000, 16), (16, 13000)])
@pytest.mark.parametrize("K", [1, 7, 8, 9, 100])
def test_large_tiles(M, N, K):
    """64 x 64, 128 x 16 and 16 x 128 tiles at the edges of their K blocks of 8 and 16."""
    tc, fp32 = binding.cc_lr_selftest_gemm(M, N, K, 2, seed=M + N + K)
    assert 0 <= fp32 < 2e-5
