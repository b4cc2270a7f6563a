"""The FP64 tensor-core GEMM on operands whose entries span many orders of magnitude within a row, the large entries of
one operand meeting the small ones of the other, and the imaginary parts lying far below the real ones.
The sizes take every way to the direct sums: a thread, a warp or the block per entry, with K of the comparison split or not.

Bound (the library divides by it, so the limit here is 1): that of FP64 sums in any order, for the real and the
imaginary part by itself.  Each part of a complex product of K terms is a sum of 2 K real products, with
one rounding per fused multiply-add, so it is off by at most 2 K u sum |terms|; alpha and the addition to C add
a few u.
"""
import pytest

from paper_2604_12914_gb300 import binding


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", [(1, 1, 3), (33, 17, 16), (129, 33, 90), (260, 70, 130), (40, 130, 700), (300, 10, 2100),
                                   (7, 7, 5000), (5000, 130, 40), (20000, 16, 24)])
@pytest.mark.parametrize("spread", [0.0, 8.0, 30.0, 60.0, 300.0])
def test_f64_gemm_of_graded_operands(M, N, K, spread):
    for layout in (32, 35, 47):  # A [K][M], B [K][N]; A [M][K], B [N][K]; those with C [N][M] and a complex alpha
        err, nans = binding.cc_lr_selftest_f64gemm(M, N, K, layout, spread=spread, seed=M + 7 * N + K)
        assert err <= 1.0, (layout, err)
        assert nans == 0


@pytest.mark.gpu
def test_captured_products_with_slices():
    """FP64 products of a size that runs on the slices, replayed from CUDA graphs (the magnitudes' sums are formed on a second
    stream, which the capture takes in): the eager results, for other inputs too.  Both are FP64-accurate and
    differ by the order of atomic additions only."""
    import torch

    from gpu_helpers import rel_err
    from paper_2604_12914_gb300.inputs import make_system, random_amplitudes
    s = make_system(8, 32, 90, seed=5, scale=0.3)
    t1, t2 = random_amplitudes(8, 32, seed=6, s1=0.05, s2=0.2)
    stream = torch.cuda.Stream()
    ctx = binding.Context(s.o, s.v, s.naux, s.eps, s.L, s.mu, t1=t1, t2=t2, prec="fp64", stream=stream.cuda_stream)
    xs = [random_amplitudes(8, 32, seed=k) for k in (7, 8)]
    eager = [(ctx.cc_lr_sigma(*x), ctx.cc_lr_sigma_T(*x)) for x in xs]
    ctx.cc_lr_set_graphs(True)
    for k in (0, 0, 0, 1, 1):
        assert rel_err(*ctx.cc_lr_sigma(*xs[k]), *eager[k][0]) < 1e-12
        assert rel_err(*ctx.cc_lr_sigma_T(*xs[k]), *eager[k][1]) < 1e-12
    captures, launches = ctx.cc_lr_graph_stats()
    assert captures == 2 and launches >= 6
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("M,N", [(129, 16), (129, 32), (20, 70)])
@pytest.mark.parametrize("K", [31, 32, 33, 32768, 33001])
def test_f64_gemm_at_chunks_and_segments_of_k(M, N, K):
    """K around a chunk (32 complex) in tiles of 32, 64 and 128 columns, and beyond what the integer sums of one launch hold
    (32768 complex), with ordinary entries and with graded ones; the library divides by the bound of each."""
    if K > 30000:
        M = min(M, 9)  # (the reference sums on the host take K per entry)
    for layout, spread in ((0, 20.0), (35, 40.0)):
        err, nans = binding.cc_lr_selftest_f64gemm(M, N, K, layout, spread=spread, seed=M + N + K)
        assert err <= 1.0, (layout, err)
        assert nans == 0
