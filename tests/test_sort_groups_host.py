"""The sort planner's blocks and register groups at their edges, on the host: the
tables give the Sec. 6.1 network's output bit for bit where the count of keys
per thread, the kind of block (one, first size beyond) or the block's size
changes, and the plan refuses and accepts the block sizes it is documented to."""

import pytest

from paper_2306_07795_gb300 import _binding as B
from test_sort_plan_host import check


@pytest.mark.parametrize("key", [B.BMMC_KEY_F32, B.BMMC_KEY_F64])
@pytest.mark.parametrize("n,b,block_log2", [(7, 0, 0), (7, 1, 0), (8, 0, 0), (9, 0, 0), (10, 0, 0),
                                            (11, 0, 0), (11, 1, 0), (13, 0, 15), (13, 0, 16),
                                            (14, 0, 16), (12, 2, 16), (3, 10, 0), (15, 0, 16)])
def test_edges(n, b, block_log2, key):
    check(n, b, key, seed=n + b, block_log2=block_log2)


@pytest.mark.parametrize("key,least", [(B.BMMC_KEY_U32, 14), (B.BMMC_KEY_I64, 15)])
def test_block_sizes(key, least):
    for n in (12, 13, 20):
        for block_log2 in (12, 13, 14, 15, 16):
            if n > 12 and block_log2 < least:
                with pytest.raises(B.BmmcError) as ei:
                    B.bmmc_sort_plan_create(n, 0, key, block_log2)
                assert ei.value.code == B.BMMC_ERR_UNSUPPORTED
                continue
            h = B.bmmc_sort_plan_create(n, 0, key, block_log2)
            e = 4 if key == B.BMMC_KEY_U32 else 8
            one = n <= 12 or e << n <= 1 << block_log2  # the block holds every key
            assert (B.bmmc_sort_plan_num_passes(h) == 1) == one
            assert B.bmmc_sort_workspace_bytes(h) == (0 if one else e << n)
            B.bmmc_sort_plan_destroy(h)


@pytest.mark.parametrize("key,e", [(B.BMMC_KEY_F32, 4), (B.BMMC_KEY_U64, 8)])
def test_workspace_of_rows(key, e):
    """Rows that fit a thread block are one pass, however many they are, and
    take no workspace; longer ones take one array."""
    for n, b in ((1, 12), (5, 20), (10, 3), (10, 10), (1, 31), (12, 1), (13, 0), (14, 6), (16, 8)):
        h = B.bmmc_sort_plan_create(n, b, key)
        one = B.bmmc_sort_plan_num_passes(h) == 1
        if n <= 10:
            assert one
        if n > 12:
            assert not one
        assert B.bmmc_sort_workspace_bytes(h) == (0 if one else e << (n + b))
        B.bmmc_sort_plan_destroy(h)


def test_fewest_passes():
    """The cuts leave a dimension for the next pass's segments."""
    for n, passes in ((16, 7), (20, 12), (24, 17)):
        h = B.bmmc_sort_plan_create(n, 0, B.BMMC_KEY_F32)
        assert B.bmmc_sort_plan_num_passes(h) <= passes
        B.bmmc_sort_plan_destroy(h)
