"""nnz-balanced SpMM (spmm_merge_kernel): every piece width, odd k, and matrices whose items end at the edges of shares, warps and tiles."""
import numpy as np
import pytest

import gen
import paper_2603_07169_b200 as b200sp
from gpu_util import assert_within, needs_plain_build, run_spmm, store, to_dev

pytestmark = pytest.mark.gpu


def matrices():
    rng = np.random.default_rng(3)
    skew = (rng.pareto(1.3, 3000) * 3).astype(np.int64).clip(0, 900)
    skew[5] = 6000                                                            # a row over several CTAs
    return {
        "skewed": skew,
        "one_share": np.array([32 - 4, 0, 0]),                                 # rows + nonzeros = 31, then exactly 32
        "share_edge": np.array([28, 0, 0, 0]),
        "cta_edge": np.concatenate([np.full(7, 31), [32]]),                    # 8 warps x 32 items, all rows ending at share ends
        "cta_edge_plus_one": np.concatenate([np.full(8, 31), [1]]),
        "one_row": np.array([5000]),
        "all_empty_but_last": np.concatenate([np.zeros(5000, np.int64), [3]]),
        "large": rng.integers(0, 60, 120_000),                                 # shares of 128 items, several to a warp
    }


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("case", sorted(matrices()))
def test_merge_spmm_against_oracle(case, dtype):
    lens = matrices()[case]
    rng = np.random.default_rng(len(case))
    n = 40_000                                                                 # too many columns for the shared-memory-B kernel
    A = gen.random_csr(len(lens), n, lens, seed=5, sort_cols=False)
    b200sp.b200sp_set_option("spmm_flat", 1)
    try:
        for k in ((50,) if case == "large" else (2, 3, 16, 33, 50, 64, 65, 100, 127, 130, 256, 300)):
            B = rng.standard_normal(n * k).astype(np.float32)
            Y0 = rng.standard_normal(A.m * k).astype(np.float32)
            Y, Y_ref, S = run_spmm(A, B, k, None, 1.0, 0.0, dtype)
            assert_within(Y, Y_ref, S, dtype, what="%s k=%d" % (case, k))
            Y, Y_ref, S = run_spmm(A, B, k, Y0, -0.5, 1.25, dtype)
            y0f = Y0 if dtype == "f32" else gen.bf16_to_f32(gen.to_bf16(Y0))
            assert_within(Y, Y_ref, S, dtype, 1.0, np.abs(1.25 * y0f.astype(np.float64)).reshape(A.m, k), what="%s k=%d ab" % (case, k))
    finally:
        b200sp.b200sp_set_option("spmm_flat", 2)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_even_rows_of_ragged_width_on_both_sides_of_the_rule(dtype):
    """k that is no multiple of a vector: by rows up to 16 columns (a group of 2 to 16 lanes per row), by shares above."""
    rng = np.random.default_rng(2)
    A = gen.random_csr(3000, 20_000, rng.integers(10, 16, 3000), seed=8)
    for k in (2, 3, 5, 7, 9, 13, 15, 17, 18, 31):
        B = rng.standard_normal(A.n * k).astype(np.float32)
        Y, Y_ref, S = run_spmm(A, B, k, None, 1.0, 0.0, dtype)
        assert_within(Y, Y_ref, S, dtype, what="k=%d" % k)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_uneven_rows_and_few_columns_by_rows(dtype):
    """Nearly even rows and a few longer ones: a lane or a few per row, rows of more than 128 by a launch of their own (aligned k)."""
    rng = np.random.default_rng(3)
    lens = rng.integers(6, 11, 200_000)
    lens[17], lens[160_000], lens[-1] = 60, 129, 140
    A = gen.random_csr(len(lens), 50_000, lens, seed=9)
    plan = b200sp.b200sp_plan_create(A.m, A.n, A.nnz, to_dev(A.row_ptr))
    stats = b200sp.b200sp_plan_info(plan)
    b200sp.b200sp_plan_destroy(plan)
    for k in (2, 3, 4, 8, 16):
        assert k > 3 or not b200sp.b200sp_spmm_by_shares(stats, k, 0.0, dtype)
        B = rng.standard_normal(A.n * k).astype(np.float32)
        Y0 = rng.standard_normal(A.m * k).astype(np.float32)
        Y, Y_ref, S = run_spmm(A, B, k, None, 1.0, 0.0, dtype)
        assert_within(Y, Y_ref, S, dtype, what="k=%d" % k)
        Y, Y_ref, S = run_spmm(A, B, k, Y0, -0.5, 1.25, dtype)
        y0f = Y0 if dtype == "f32" else gen.bf16_to_f32(gen.to_bf16(Y0))
        assert_within(Y, Y_ref, S, dtype, 1.0, np.abs(1.25 * y0f.astype(np.float64)).reshape(A.m, k), what="k=%d ab" % k)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_old_values_asked_for_ahead_belong_to_their_rows(dtype):
    """beta != 0 and no empty rows: Y's old values of a row are read when the row before it ends.  Old values that differ from row to row by
    more than the products, rows that end at the first and the last nonzero of a group of 8 and of a share, several to a group, and every
    number of loads per nonzero (k up to 256 and a second slice)."""
    lens = np.concatenate([np.arange(1, 41), np.full(200, 1), np.full(64, 8), np.full(33, 31), [700], np.full(60, 7), [1]])
    n = 30_000
    A = gen.random_csr(len(lens), n, lens, seed=17, sort_cols=False)
    rng = np.random.default_rng(4)
    b200sp.b200sp_set_option("spmm_flat", 1)
    try:
        for k in (2, 17, 33, 50, 63, 64, 100, 127, 128, 130, 256, 320):
            B = rng.standard_normal(n * k).astype(np.float32)
            Y0 = np.repeat((64 + 64 * (np.arange(A.m) % 4)).astype(np.float32), k)
            Y, Y_ref, S = run_spmm(A, B, k, Y0, 0.5, -1.0, dtype)
            assert_within(Y, Y_ref, S, dtype, 0.5, np.abs(Y0.astype(np.float64)).reshape(A.m, k), what="k=%d" % k)
    finally:
        b200sp.b200sp_set_option("spmm_flat", 2)


def test_non_finite_rows_of_b_touch_only_the_rows_that_use_them():
    """What a warp reads ahead of its last nonzero (row 0 of B) is never multiplied."""
    n, k = 9000, 64
    lens = np.full(77, 5)
    lens[::4] = 0
    A = gen.random_csr(len(lens), n, lens, seed=1)
    A.col_idx[:] = np.maximum(A.col_idx, 1)
    B = np.ones(n * k, np.float32)
    B[:k] = np.inf
    b200sp.b200sp_set_option("spmm_flat", 1)
    try:
        Y, Y_ref, S = run_spmm(A, B, k, None, 1.0, 0.0, "f32")
        assert np.isfinite(Y).all()
        assert_within(Y, Y_ref, S, "f32")
    finally:
        b200sp.b200sp_set_option("spmm_flat", 2)


@needs_plain_build
@pytest.mark.parametrize("dtype,ks", [("f32", (63, 127, 256, 512)), ("bf16", (63, 66, 127, 256, 264, 512))])
def test_old_values_cost_no_more_than_their_bytes_and_a_wait(dtype, ks):
    """beta != 0 against beta == 0, same call: Y is read once more, and a form without registers for what it reads ahead spills.  1.3 times
    at most with 20 nonzeros a row; k = 264 BF16 took 2.1 times as long when two loads of eight columns read ahead as well."""
    import torch
    lens = np.random.default_rng(5).integers(2, 40, 70_000)
    n = len(lens)
    A = gen.random_csr(n, n, lens, seed=6, sort_cols=False)
    d = [to_dev(a) for a in (A.row_ptr, A.col_idx, store(A.vals, dtype))]
    b200sp.b200sp_set_option("spmm_flat", 1)
    try:
        for k in ks:
            B, Y = (torch.zeros(n * k, dtype=torch.float32 if dtype == "f32" else torch.int16, device="cuda:0") for _ in range(2))
            times = []
            for beta in (0.0, 0.5):
                best = 1e9
                for _ in range(8):
                    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    start.record()
                    for _ in range(4):
                        b200sp.spmm_csr(n, n, A.nnz, k, d[0], d[1], d[2], B, Y, 1.0, beta, dtype)
                    end.record()
                    torch.cuda.synchronize()
                    best = min(best, start.elapsed_time(end))
                times.append(best)
            assert times[1] < 1.4 * times[0], "k=%d: %.3f ms with beta == 0, %.3f ms with beta != 0" % (k, times[0] / 4, times[1] / 4)
    finally:
        b200sp.b200sp_set_option("spmm_flat", 2)
        b200sp.b200sp_cache_clear()


@pytest.mark.parametrize("dtype,k", [("bf16", 100), ("bf16", 130), ("bf16", 256), ("f32", 66), ("f32", 256)])
def test_several_shares_to_a_warp(dtype, k):
    """Shares of 128 items, several to a warp, at widths that stay by shares on a matrix of this size."""
    lens = matrices()["large"]
    rng = np.random.default_rng(k)
    n = 40_000
    A = gen.random_csr(len(lens), n, lens, seed=5, sort_cols=False)
    stats = dict(m=A.m, n=n, nnz=A.nnz, min_row_len=0, max_row_len=59, bin_rows=[2000, 8000, 56_000, 54_000, 0, 0], bin_nnz=[0, 20_000, 1_000_000, A.nnz - 1_020_000, 0, 0])
    b200sp.b200sp_set_option("spmm_flat", 1)
    try:
        assert not any(b200sp.b200sp_spmm_by_bundles(stats, k, beta, dtype) for beta in (0.0, 1.25))
        B, Y0 = rng.standard_normal(n * k).astype(np.float32), rng.standard_normal(A.m * k).astype(np.float32)
        Y, Y_ref, S = run_spmm(A, B, k, None, 1.0, 0.0, dtype)
        assert_within(Y, Y_ref, S, dtype)
        Y, Y_ref, S = run_spmm(A, B, k, Y0, -0.5, 1.25, dtype)
        y0f = Y0 if dtype == "f32" else gen.bf16_to_f32(gen.to_bf16(Y0))
        assert_within(Y, Y_ref, S, dtype, 1.0, np.abs(1.25 * y0f.astype(np.float64)).reshape(A.m, k))
    finally:
        b200sp.b200sp_set_option("spmm_flat", 2)
