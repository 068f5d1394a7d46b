"""Split points of the plan pass as it takes them from the rows, on the host (no GPU needed), against the search that defines them."""
import numpy as np
import pytest

import paper_2603_07169_b200 as b200sp


def searched(row_ptr, nnz, items):
    """First row whose end lies behind the diagonal, within what m and nnz allow."""
    m = len(row_ptr) - 1
    d = np.minimum(np.arange((m + nnz + items - 1) // items + 1, dtype=np.int64) * items, m + nnz)
    ends = row_ptr[1:].astype(np.int64) + np.arange(1, m + 1)
    return np.clip(np.searchsorted(ends, d, side="right"), np.maximum(d - nnz, 0), np.minimum(d, m))


def offsets(lens, start=0):
    return (start + np.concatenate([[0], np.cumsum(lens)])).astype(np.int64)


def split_points(row_ptr, nnz, items):
    m = len(row_ptr) - 1
    out = np.full((m + nnz + items - 1) // items + 1, -7, np.int32)
    b200sp.b200sp_split_points(m, nnz, row_ptr.astype(np.int32), items, out)
    return out.astype(np.int64)


RNG = np.random.default_rng(0)
MIXED = RNG.choice([0, 0, 1, 5, 31, 130, 3000], 5000)
CASES = {                                                        # offsets, nnz
    "mixed": (offsets(MIXED), int(MIXED.sum())),
    "one_row": (offsets([70_000]), 70_000),
    "empty_but_one": (offsets(np.r_[np.zeros(900), 5, np.zeros(400)]), 5),
    "no_nonzeros": (offsets(np.zeros(300)), 0),
    "largest_with_shares": (offsets(np.r_[np.full(1000, 2000), np.full(7, 7), (1 << 23) - 1008 - 2_000_049]), (1 << 23) - 1008),
    # not what a plan asks for: rows of a larger matrix with their offsets as they are, a count of nonzeros that is not the last offset
    "offset": (offsets(MIXED, 100_000), int(MIXED.sum())),
    "offset_past_2^29": (offsets(MIXED, 3 << 29), int(MIXED.sum())),
    "count_too_small": (offsets(MIXED), int(MIXED.sum()) // 3),
    "count_too_large": (offsets(MIXED), int(MIXED.sum()) * 2),
    "negative": (offsets(MIXED, -100_000), int(MIXED.sum())),
}


@pytest.mark.parametrize("items", [32, 40, 56, 120, 128, 1024, 2048, 4096])
@pytest.mark.parametrize("case", sorted(CASES))
def test_split_points(case, items):
    row_ptr, nnz = CASES[case]
    m = len(row_ptr) - 1
    out = split_points(row_ptr, nnz, items)
    assert np.array_equal(out, searched(row_ptr, nnz, items))
    nonzero = np.minimum(np.arange(len(out), dtype=np.int64) * items, m + nnz) - out
    assert nonzero.min() >= 0 and nonzero.max() <= nnz and out.min() >= 0 and out.max() <= m


@pytest.mark.parametrize("items", [1024, 4096])
def test_tiles_up_to_the_largest_sizes(items):
    """m + nnz just below 2^32: item numbers in all of 32 bits."""
    m, nnz = (1 << 31) // 1024, (1 << 31) - 1
    row_ptr = np.minimum(np.arange(m + 1, dtype=np.int64) * 1024, nnz)
    assert np.array_equal(split_points(row_ptr, nnz, items), searched(row_ptr, nnz, items))


def test_refused():
    for m, nnz, items in ((4, 10, 16), (4, 10, 136), (4, 1 << 29, 40), (-1, 0, 32)):
        assert b200sp.lib().b200sp_split_points(m, nnz, np.zeros(8, np.int32).ctypes.data, items, np.zeros(8, np.int32).ctypes.data) == 1
