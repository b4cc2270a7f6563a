"""Tensor-core GEMMs by pairs of CTAs (256-row tiles) at the edges of their tiles, splits and accumulators."""
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


@pytest.mark.parametrize("M,N,K", [
    (256, 33, 31),       # one K chunk less a complex entry
    (255, 40, 32),       # one full chunk
    (100, 300, 48),      # second CTA without rows; half a chunk at the end
    (385, 70, 49),       # ... and less than a quarter of one
    (5200, 260, 40),     # several units per pair: accumulators and slots wrap at any phase
])
@pytest.mark.parametrize("layout", [0, 3])
def test_f64_pair_gemm_within_bound(M, N, K, layout):
    """FP64 GEMM from exact slices against extended precision; the library divides by the bound that the tests of the
    slices derive, so the limit is 1."""
    from paper_2604_12914_gb300 import binding
    err, nans = binding.cc_lr_selftest_f64gemm(M, N, K, layout, spread=20.0, seed=M + 7 * N + K)
    assert err <= 1.0, err
    assert nans == 0
