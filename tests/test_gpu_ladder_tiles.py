"""sigma and its transpose at virtual spaces on both sides of the ladder's tile and group edges (formation
tiles of 128 rows by 64 to 128 columns, of which only those with an entry b > a are computed, in groups of 8 to 64
values of a; K rows padded to whole 128-byte blocks from 64 on), against the oracle.

Tolerances are those of the existing parity tests of each mode.
"""
import pytest

from gpu_helpers import gpu_context, oracle_sigma, oracle_sigma_T, rel_err
from paper_2604_12914_gb300.inputs import make_system, random_amplitudes


@pytest.mark.gpu
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("3xtf32", 5e-5), ("bf16x3", 3e-4), ("tf32", 3e-3)])
@pytest.mark.parametrize("v,naux", [(31, 63), (33, 64), (40, 65), (47, 70)])
def test_sigma_at_tile_edges(prec, tol, v, naux):
    s = make_system(3, v, naux, seed=v, scale=0.3)
    t1, t2 = random_amplitudes(3, v, seed=v + 1, s1=0.05, s2=0.2)
    x1, x2 = random_amplitudes(3, v, seed=v + 2)
    ctx = gpu_context(s, t1=t1, t2=t2, prec=prec)
    g1, g2 = ctx.cc_lr_sigma(x1, x2)
    r1, r2 = oracle_sigma(s, t1, t2, x1, x2)
    assert rel_err(g1, g2, r1, r2) < tol
    z1, z2 = ctx.cc_lr_sigma_T(x1, x2)
    q1, q2 = oracle_sigma_T(s, t1, t2, x1, x2)
    assert rel_err(z1, z2, q1, q2) < tol
    ctx.close()
