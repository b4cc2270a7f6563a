"""FP64 sigma and its transpose with the slices of L~_vv made in chunks (budgeted contexts keep none): the oracle's results, and
no more memory than the chunks.  The tolerance is the FP64 mode's parity bound."""
import pytest

from gpu_helpers import oracle_sigma, oracle_sigma_T, rel_err
from paper_2604_12914_gb300 import binding
from paper_2604_12914_gb300.inputs import make_system, random_amplitudes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("v,naux", [(40, 65), (47, 70)])
def test_ladder_slices_in_chunks(v, naux):
    s = make_system(4, v, naux, seed=v, scale=0.3)
    t1, t2 = random_amplitudes(4, v, seed=v + 1, s1=0.05, s2=0.2)
    x1, x2 = random_amplitudes(4, v, seed=v + 2)
    r, q = oracle_sigma(s, t1, t2, x1, x2), oracle_sigma_T(s, t1, t2, x1, x2)
    row = 36 * naux  # bytes of a row's slices; a column's are twice that
    for cap in (2 << 30, 700 * row, 131 * row):  # whole, in a few chunks, in many that end within a tile
        ctx = binding.Context(s.o, s.v, s.naux, s.eps, s.L, s.mu, t1=t1, t2=t2, prec="fp64", hbm_budget=8 << 30)
        binding.cc_lr_selftest_f64_operand_cap(ctx, cap)
        assert rel_err(*ctx.cc_lr_sigma(x1, x2), *r) < 1e-10
        assert rel_err(*ctx.cc_lr_sigma_T(x1, x2), *q) < 1e-10
        ctx.close()


def test_peak_memory_follows_the_limit():
    o, v, naux = 3, 64, 600
    s = make_system(o, v, naux, seed=1, scale=0.3)
    x = random_amplitudes(o, v, seed=2)
    peak = []
    for cap in (2 << 30, 4 << 20):
        ctx = binding.Context(s.o, s.v, s.naux, s.eps, s.L, s.mu, prec="fp64", hbm_budget=8 << 30)
        binding.cc_lr_selftest_f64_operand_cap(ctx, cap)
        ctx.cc_lr_sigma(*x)
        peak.append(ctx.cc_lr_memory()[1])
        ctx.close()
    whole = 36 * naux * v * v + 72 * naux * 16 * v  # the rows of all of L~_vv, the columns of a group of 16
    assert peak[0] - peak[1] > whole
