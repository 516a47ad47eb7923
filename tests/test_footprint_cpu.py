"""kh_footprint's bound on the host (no GPU): graphs that cannot have a node whose
union is split count no part slots, the others do."""
import pytest

from paper_2112_06154_gb300 import build as B
from paper_2112_06154_gb300 import khcore as K


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()
    K.load()


# a node is split on graphs with one of more than 2048 neighbours: 2050 nodes and twice
# 2049 entries at least
@pytest.mark.parametrize("n,nnz,slots", [(2049, 2049 * 2048, False), (2049, 4098, False), (2050, 4097, False),
                                         (2050, 4098, True), (60000, 4097, False), (60000, 600000, True)])
def test_part_slots_are_counted_where_a_split_is_possible(n, nnz, slots):
    M = 600
    bare = K.kh_footprint(n, 0, 2, M)[1]
    extra = K.kh_footprint(n, nnz, 2, M)[1] - bare
    want = 4 * nnz  # the columns
    if slots:
        want += nnz // 341 * (4 * M + 32) + 4 * n
    assert extra == want
