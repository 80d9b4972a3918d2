"""The roofline arithmetic of bench.py: operations and bytes of the executed form
(products between parents and between blocks), on counts that can be written
down, and a fraction above 1 reported as an error."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

NONE = dict(parent_pairs=0, block_pairs=0, parent_fwd=0, parent_inv=0, block_fwd=0, block_inv=0)


@pytest.mark.parametrize("N", [8, 16])
def test_executed_work(N):
    # one octree level of 4^3 blocks: 2^3 parents, each with every parent
    w = dict(NONE, parent_pairs=64, parent_fwd=8, parent_inv=8)
    padded, cells = (4 * N) * (4 * N) * (2 * N + 1), (2 * N) ** 3   # of a parent
    x = bench.executed_work(w, N, 4)
    assert x["mac_flops"] == 64 * padded * 8
    # half a padded spectrum: the axis that the product kernel transforms is not padded in memory
    assert x["fwd_bytes"] == x["inv_bytes"] == 8 * (cells * 4 + padded // 2 * 8)
    x = bench.executed_work(w, N, 8)
    assert x["mac_flops"] == 64 * padded * 6
    assert x["fwd_bytes"] == 8 * (cells * 8 + padded // 2 * 16 + (padded // 2 + padded) * 16)
    # block by block
    w = dict(NONE, block_pairs=27, block_fwd=3, block_inv=2)
    padded = (2 * N) * (2 * N) * (N + 1)
    for rs in (4, 8):
        x = bench.executed_work(w, N, rs)
        assert x["mac_flops"] == 27 * padded * 8
        assert x["fwd_bytes"] == 3 * (N ** 3 * rs + padded * 2 * rs)
        assert x["inv_bytes"] == 2 * (N ** 3 * rs + padded * 2 * rs)


def test_fraction_above_one_is_an_error():
    errors = []
    assert bench.fraction(3.0, 4.0, "a", errors) == 0.75 and errors == []
    assert bench.fraction(5.43, 1.0, "b", errors) is None and len(errors) == 1 and "b" in errors[0]
