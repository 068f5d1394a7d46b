"""The rule that sends SpMM to the nnz-balanced kernel, on the host (no GPU needed)."""
import pytest

import paper_2603_07169_b200 as b200sp


def info(m, n, bin_rows, bin_nnz, longest):
    return dict(m=m, n=n, nnz=sum(bin_nnz), min_row_len=0, max_row_len=longest, bin_rows=bin_rows, bin_nnz=bin_nnz)


@pytest.mark.parametrize("dtype,size", [("f32", 4), ("bf16", 2)])
def test_rows_of_b_too_wide_for_32_bit_offsets_go_by_rows(dtype, size):
    """The kernel steps over a row of B by a 32-bit number of bytes and counts columns up to a slice (512) past k in 32 bits."""
    uneven = info(2, 2, [1, 1, 0, 0, 0, 0], [0, 2, 0, 0, 0, 0], 2)
    even = info(2, 2, [0, 2, 0, 0, 0, 0], [0, 4, 0, 0, 0, 0], 2)
    last = (2**31 - 1 - 2048) // size
    assert last * size < 2**31 and last + 512 < 2**31
    assert b200sp.b200sp_spmm_by_shares(uneven, 64, dtype) and b200sp.b200sp_spmm_by_shares(uneven, last, dtype)
    for k in (last + 1, 2**31 // size, 2**31 // size + 1, 2**31 // size + 64, 2**31 - 8, 2**31 - 1):
        assert not b200sp.b200sp_spmm_by_shares(uneven, k, dtype) and not b200sp.b200sp_spmm_by_shares(even, k, dtype), k
