"""One-pass tensor-core GEMM by pairs of CTAs (256-row tiles) at the edges of its tiles, splits and accumulators."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    (129, 128, 64),      # one row in the second CTA's half
    (256, 64, 40),       # one 128-wide tile
    (257, 150, 33),      # second pair with one row, ragged last column tile and K block
    (384, 129, 17),      # pair whose second CTA has no rows
    (512, 80, 9000),     # 160 columns, K splits added atomically
    (20100, 256, 48),    # several units per pair: both accumulators and the ring wrap
    (2000, 1100, 700),   # many column tiles, six ring slots wrap at any phase
])
def test_pair_gemm_against_fp64(M, N, K):
    from paper_2604_12914_gb300 import binding
    tc, _ = binding.cc_lr_selftest_gemm(M, N, K, 1, seed=M + N + K)
    assert tc >= 0, "tensor-core path not taken"
    # both operands keep 10 mantissa bits, cut off: each product is off by less than 2^-9 of itself, one way or the
    # other, so a sum of K of them by less than 2^-9 of the root of K products, which max |C| is above
    assert tc < 2.0 ** -8
