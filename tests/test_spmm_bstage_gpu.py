"""SpMM with a slice of B in shared memory: two 16-byte pieces per lane (calls with a step for every warp) and one, the re-ordered blocks of
64-byte slices, a last block, a last CTA of the copy of A and a last slice that are not full, and one plan used with both."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2603_07169_b200 as b200sp
from gpu_util import assert_within, empty_out, run_spmm, store, to_dev, to_host

pytestmark = pytest.mark.gpu


def lengths(m, n, seed):
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, 45, m)
    lens[:6] = [0, 1, 1024, 1025, 700, 129]       # up to kLongRow, above it, and several blocks of a lane's chain
    return np.minimum(lens, n)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n,m,k", [(2048, 3001, 900), (2048, 3008, 1032), (2048, 3024, 904), (1700, 2003, 520), (1700, 2000, 1048), (3300, 3015, 888), (300, 1999, 1024),
                                   (2048, 9999, 1000), (2048, 10003, 904)])       # the last two: blocks re-ordered
def test_against_oracle(n, m, k, dtype):
    rng = np.random.default_rng(m + k)
    if dtype == "bf16":
        k *= 2
    A = gen.random_csr(m, n, lengths(m, n, m), seed=n, sort_cols=False)
    B = rng.standard_normal(n * k).astype(np.float32)
    Y, Y_ref, S = run_spmm(A, B, k, None, 1.0, 0.0, dtype)
    assert_within(Y, Y_ref, S, dtype, what="n=%d m=%d k=%d" % (n, m, k))
    Y0 = rng.standard_normal(m * k).astype(np.float32)
    Y, Y_ref, S = run_spmm(A, B, k, Y0, -0.5, 1.25, dtype)
    y0f = Y0 if dtype == "f32" else gen.bf16_to_f32(gen.to_bf16(Y0))
    assert_within(Y, Y_ref, S, dtype, 1.0, np.abs(1.25 * y0f.astype(np.float64)).reshape(m, k), what="n=%d m=%d k=%d ab" % (n, m, k))
    b200sp.b200sp_check()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n,m,k", [(2048, 9001, 904), (2048, 9999, 1000), (1700, 9003, 1048)])
def test_old_values_of_y_with_two_pieces(n, m, k, dtype):
    """beta != 0 with steps enough for two pieces per lane: the old values are loaded ahead, past the last column and row as zeros."""
    rng = np.random.default_rng(m)
    if dtype == "bf16":
        k *= 2
    A = gen.random_csr(m, n, lengths(m, n, m) // 3, seed=n, sort_cols=False)
    B, Y0 = rng.standard_normal(n * k).astype(np.float32), rng.standard_normal(m * k).astype(np.float32)
    Y, Y_ref, S = run_spmm(A, B, k, Y0, -0.5, 1.25, dtype)
    y0f = Y0 if dtype == "f32" else gen.bf16_to_f32(gen.to_bf16(Y0))
    assert_within(Y, Y_ref, S, dtype, 1.0, np.abs(1.25 * y0f.astype(np.float64)).reshape(m, k), what="n=%d m=%d k=%d" % (n, m, k))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_rows_in_columns_of_one_parity(dtype):
    """All of a row's columns even, or all odd, in every mixture inside a block: the re-ordering at its extremes."""
    rng = np.random.default_rng(4)
    m, n, k = 10003, 2048, 928 if dtype == "f32" else 1856
    A = gen.random_csr(m, n, rng.integers(10, 14, m), seed=9, sort_cols=False, allow_dup=True)
    rows = np.repeat(np.arange(m), np.diff(A.row_ptr))
    A.col_idx[:] = (A.col_idx & ~1) | (rng.random(m) < 0.3)[rows]
    B = rng.standard_normal(n * k).astype(np.float32)
    Y, Y_ref, S = run_spmm(A, B, k, None, 1.0, 0.0, dtype)
    assert_within(Y, Y_ref, S, dtype, what="one parity")


def test_one_plan_with_narrow_and_wide_products():
    """Narrow k takes one piece per lane, wide k two: each has its own order of the rows, kept in the plan."""
    rng = np.random.default_rng(8)
    m, n = 3001, 2048
    A = gen.random_csr(m, n, lengths(m, n, 3), seed=7)
    d_rp, d_ci, d_va = to_dev(A.row_ptr), to_dev(A.col_idx), to_dev(store(A.vals, "f32"))
    plan = b200sp.b200sp_plan_create(m, n, A.nnz, d_rp)
    for k in (64, 1024, 64, 512):
        B = rng.standard_normal(n * k).astype(np.float32)
        d_Y = empty_out(m * k, "f32")
        b200sp.b200sp_spmm(plan, k, d_ci, d_va, to_dev(B), d_Y, 1.0, 0.0, "f32")
        torch.cuda.synchronize()
        Y_ref, S = oracle.spmm_csr(m, n, k, A.row_ptr, A.col_idx, A.vals, B, None, 1.0, 0.0, "f32", nthreads=oracle.max_threads())
        assert_within(to_host(d_Y, "f32").reshape(m, k), np.asarray(Y_ref).reshape(m, k), np.asarray(S).reshape(m, k), "f32", what="k=%d" % k)
    b200sp.b200sp_plan_destroy(plan)
