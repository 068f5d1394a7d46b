"""SpMV on both sides of the sub-warp rule, and rows cut by tile boundaries at the edges of the carry fix-up's groups of 16."""
import numpy as np
import pytest
import torch

import gen
import paper_2603_07169_b200 as b200sp
from gpu_util import assert_within, run_spmv, to_dev

pytestmark = pytest.mark.gpu


def check(A, dtype, what):
    rng = np.random.default_rng(A.m)
    x, y0 = rng.standard_normal(A.n).astype(np.float32), rng.standard_normal(A.m).astype(np.float32)
    y, y_ref, S = run_spmv(A, x, None, 1.0, 0.0, dtype)
    assert_within(y, y_ref, S, dtype, what=what)
    y, y_ref, S = run_spmv(A, x, y0, -0.5, 1.25, dtype)
    y0f = y0 if dtype == "f32" else gen.bf16_to_f32(gen.to_bf16(y0))
    assert_within(y, y_ref, S, dtype, 1.0, np.abs(1.25 * y0f.astype(np.float64)), what=what)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("longest,kernel", [(40, 3), (160, 3), (161, 0), (2000, 0)])
def test_sub_warps_only_while_no_lane_has_a_long_chain(longest, kernel, dtype):
    lens = np.full(3000, 9)                       # four lanes to a row
    lens[1234] = longest
    A = gen.random_csr(len(lens), 5000, lens, seed=longest)
    plan = b200sp.b200sp_plan_create(A.m, A.n, A.nnz, to_dev(A.row_ptr))
    assert b200sp.b200sp_plan_info(plan)["spmv_kernel"] == kernel
    b200sp.b200sp_plan_destroy(plan)
    check(A, dtype, "longest=%d" % longest)


def test_tile_size_by_the_rule_and_as_set():
    """1024 items below 12 million, 2048 from there on, unless the caller sets a size; 0 gives the choice back."""
    def items(m, nnz):
        row_ptr = torch.clamp(torch.arange(m + 1, device="cuda") * 8, max=nnz).int()
        plan = b200sp.b200sp_plan_create(m, 1000, nnz, row_ptr)
        found = b200sp.b200sp_plan_info(plan)["spmv_tile_items"]
        b200sp.b200sp_plan_destroy(plan)
        return found

    below, above = (1_500_000, 10_499_999), (1_500_000, 10_500_000)
    b200sp.b200sp_set_option("merge_items", 0)
    try:
        assert (items(*below), items(*above)) == (1024, 2048)
        for size in (2048, 4096, 1024):
            b200sp.b200sp_set_option("merge_items", size)
            assert (items(*below), items(*above)) == (size, size)
    finally:
        b200sp.b200sp_set_option("merge_items", 0)
    assert (items(*below), items(*above)) == (1024, 2048)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("tiles", [1, 2, 15, 16, 17, 32, 33, 40])
def test_rows_cut_by_tile_boundaries(tiles, dtype):
    """Rows over `tiles` tiles of 1024 items that begin and end at a boundary, one item before it and one after."""
    for off in (-1, 0, 1):
        for end in (-1, 0, 1):
            lens = np.concatenate([np.full(64, 63), [1024 * tiles - 1 + end - off], np.full(100, 30)])
            lens[0] += off                        # 64 x (63 + 1) = 4 x 1024 items before the row
            check(gen.random_csr(len(lens), 60_000, lens, seed=tiles, sort_cols=False), dtype, "tiles=%d off=%d end=%d" % (tiles, off, end))
