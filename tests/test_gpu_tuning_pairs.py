"""The tuning record says which shapes run by pairs of CTAs: the kernels differ where tile width, splits and band do not."""
import pytest

from paper_2604_12914_gb300 import binding
from paper_2604_12914_gb300.inputs import make_system, random_amplitudes


@pytest.mark.gpu
def test_record_tells_pairs_from_single_ctas():
    o, v = 7, 66
    s = make_system(o, v, 200, seed=3)
    ctx = binding.Context(s.o, s.v, s.naux, s.eps, s.L, s.mu, prec="tf32")
    ctx.cc_lr_sigma(*random_amplitudes(o, v, seed=3))
    rows, pairs = ctx.cc_lr_gemm_tuning(), ctx.cc_lr_gemm_tuning_pairs()
    assert len(pairs) == len(rows) > 0
    # a pair's tile has 256 rows and a width that divides by 32; up to 128 rows and 127 real columns stay with single CTAs
    for row, pair in zip(rows, pairs):
        assert not pair or (row["M"] > 128 and row["N"] >= 128 and row["BN"] % 32 == 0)
        if pair:
            assert row["band"] <= -(-row["M"] // 256)
    assert any(pairs) and not all(pairs)
    ctx.close()
