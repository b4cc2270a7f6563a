"""The tensor-core ladder packs the (e < f) pairs of a large virtual space in chunks; each chunk reads the tiles of the formed
block that hold one of its pairs, and no others.  (No GPU: the rule is host arithmetic as well.)
"""
import pytest

from paper_2604_12914_gb300 import binding, build


@pytest.fixture(scope="module", autouse=True)
def lib():
    return binding.load(build.build())


@pytest.mark.parametrize("v", [2, 15, 16, 17, 33, 64, 97, 100])
@pytest.mark.parametrize("nq", [1, 7, 64, 72, 104, 800, 10000])
def test_chunks_read_their_own_tiles(v, nq):
    pairs = v * (v - 1) // 2
    for q0 in range(0, pairs, nq):
        n = min(nq, pairs - q0)
        read, held, missed = binding.cc_lr_selftest_pack_tiles(v, q0, n)
        assert missed == 0
        assert read == held or n < v


def test_two_chunks_read_little_more_than_one():
    v = 480
    pairs = v * (v - 1) // 2
    whole, _, _ = binding.cc_lr_selftest_pack_tiles(v, 0, pairs)
    assert whole == 30 * 31 // 2
    half = (pairs + 15) // 16 * 8
    parts = [binding.cc_lr_selftest_pack_tiles(v, q0, min(half, pairs - q0))[0] for q0 in (0, half)]
    assert sum(parts) <= whole + 30  # (a row of tiles is shared)
