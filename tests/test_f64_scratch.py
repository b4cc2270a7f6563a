"""The room that the FP64 tensor-core products claim for their sums before a call's first product serves every later
one of that call: it grows with the rows and with the columns, so a smaller block never needs more than the
largest.  (No GPU: the size is host arithmetic.)
"""
import pytest

from paper_2604_12914_gb300 import binding, build


@pytest.fixture(scope="module", autouse=True)
def lib():
    return binding.load(build.build())


@pytest.mark.parametrize("v", [17, 31, 40, 77, 110, 160, 296, 480])
def test_ladder_groups_fit_the_first_groups_room(v):
    group, po = 16, max(1, (v // 6) * (v // 6 - 1) // 2)
    pairs = lambda a: a * v - a * (a + 1) // 2  # noqa: E731
    need = binding.cc_lr_selftest_f64_scratch
    first = need(v * v, min(group, v) * v), need(pairs(min(group, v)), po), need(po, v * (v - 1) // 2)
    for a0 in range(0, v - 1, group):
        a1 = min(v, a0 + group)
        assert need((v - a0) * v, (a1 - a0) * v) <= first[0]
        assert need(max(1, pairs(a1) - pairs(a0)), po) <= first[1]
    assert max(first) <= 256 << 20


def test_grows_with_rows_and_columns():
    sizes = [1, 15, 16, 17, 32, 33, 64, 65, 127, 128, 129, 500, 1000, 4864, 9728, 9729, 50000, 300000, 1000000]
    need = {(m, n): binding.cc_lr_selftest_f64_scratch(m, n) for m in sizes for n in sizes}
    for i, m in enumerate(sizes):
        for j, n in enumerate(sizes):
            if i:
                assert need[sizes[i - 1], n] <= need[m, n]
            if j:
                assert need[m, sizes[j - 1]] <= need[m, n]
