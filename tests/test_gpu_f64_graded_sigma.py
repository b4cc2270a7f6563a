"""FP64 sigma and its transpose, entry by entry, with virtual orbitals scaled over many orders of magnitude: integrals by 2^c_a for
every virtual index a, amplitudes by 2^-c_a, c from 0 to 20.  The terms of most contractions are of one size then, while the
largest entries of one operand's rows meet the smallest ones of the other's.

Of the unique entries of each result 99 in 100 have to agree with the oracle to 1e-9 of themselves: a few thousand roundings of
2^-53, with room for sums that cancel a thousandfold.  Entries lost below the largest of their row or column
are off by up to 2^-24, entries summed from wrong operands by all of themselves.
"""
import numpy as np
import pytest

from gpu_helpers import gpu_context, oracle_sigma, oracle_sigma_T
from paper_2604_12914_gb300.inputs import make_system, random_amplitudes


def _amplitudes(o, v, seed, f):
    a1, a2 = random_amplitudes(o, v, seed=seed, s1=0.05, s2=0.2)
    return a1 / f, a2 / (f[:, None] * f)


@pytest.mark.gpu
@pytest.mark.parametrize("o,v,naux", [(8, 32, 90), (5, 41, 77), (9, 50, 120)])
def test_sigma_of_scaled_orbitals(o, v, naux):
    s = make_system(o, v, naux, seed=o + v, scale=0.3)
    f = np.exp2(np.floor(np.linspace(0.0, 20.0, v)))
    full = np.concatenate([np.ones(o), f])
    s.L = s.L * (full[:, None] * full)
    t1, t2 = _amplitudes(o, v, v + 1, f)
    x1, x2 = _amplitudes(o, v, v + 2, f)
    i, j = np.triu_indices(o, 1)
    a, b = np.triu_indices(v, 1)
    ctx = gpu_context(s, t1=t1, t2=t2, prec="fp64")
    for got, ref in ((ctx.cc_lr_sigma(x1, x2), oracle_sigma(s, t1, t2, x1, x2)),
                     (ctx.cc_lr_sigma_T(x1, x2), oracle_sigma_T(s, t1, t2, x1, x2))):
        for g, r in ((got[0], ref[0]), (got[1][i, j][:, a, b], ref[1][i, j][:, a, b])):
            rel = np.abs(g - r) / np.abs(r)
            print(f"{rel.size} entries, relative error: median {np.median(rel):.1e}, 99 % {np.quantile(rel, 0.99):.1e}, "
                  f"largest {rel.max():.1e}")
            assert np.quantile(rel, 0.99) < 1e-9
    ctx.close()
