"""What the ground-state calls keep: vectors of at most 64 MB outside budgeted contexts, and nothing in budgeted ones, where a
call that finds no memory gives back its own as well."""
import pytest

from paper_2604_12914_gb300 import binding
from paper_2604_12914_gb300.inputs import make_system, random_amplitudes

pytestmark = pytest.mark.gpu


def _vector_bytes(o, v):
    return 16 * (o * v + o * (o - 1) // 2 * (v * (v - 1) // 2))


def test_solve_keeps_no_large_vectors():
    o, v = 16, 270
    assert _vector_bytes(o, v) > 64 << 20
    s = make_system(o, v, 6, seed=3, scale=0.01)
    ctx = binding.Context(s.o, s.v, s.naux, s.eps, s.L, s.mu, prec="tf32")
    ctx.cc_lr_ccsd_residual(*random_amplitudes(o, v, seed=4, s1=1e-3, s2=1e-3))
    held = ctx.cc_lr_memory()[0]
    ctx.cc_lr_ccsd(tol=1e-9, max_iterations=2, allow_noconv=True)
    assert ctx.cc_lr_memory()[0] - held < 1 << 20
    ctx.close()


def test_failed_residual_gives_its_buffers_back():
    o, v = 12, 60
    s = make_system(o, v, 40, seed=3, scale=0.05)
    x = random_amplitudes(o, v, seed=5)

    def after_sigma(budget):
        ctx = binding.Context(s.o, s.v, s.naux, s.eps, s.L, s.mu, prec="tf32", hbm_budget=budget)
        ctx.cc_lr_sigma(*x)
        return ctx

    ctx = after_sigma(1 << 36)
    peak = ctx.cc_lr_memory()[1]
    ctx.close()
    ctx = after_sigma(peak)
    held = ctx.cc_lr_memory()[0]
    with pytest.raises(binding.CclrError) as e:
        ctx.cc_lr_ccsd_residual(*random_amplitudes(o, v, seed=4, s1=1e-3, s2=1e-2))
    assert e.value.status == binding.CCLR_ENOMEM
    # the packed <ij||ab> stays (one vector's bytes); the call's own five vectors and its intermediates do not
    assert ctx.cc_lr_memory()[0] - held < 1.5 * _vector_bytes(o, v)
    ctx.close()
