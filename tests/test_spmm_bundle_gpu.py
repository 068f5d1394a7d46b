"""SpMM with rows of about equal length side by side (spmm_bundle_kernel): every width and store, rows and empty rows at the ends of regions and tiles."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2603_07169_b200 as b200sp
from gpu_util import assert_within, empty_out, needs_plain_build, run_spmm, store, to_dev, to_host

pytestmark = pytest.mark.gpu

WIDTHS = {"f32": (4, 16, 20, 32, 36, 64, 100, 128, 17, 33, 63), "bf16": (8, 24, 32, 40, 64, 72, 128, 17, 33, 65, 127, 18, 50, 126)}


def lengths(case):
    rng = np.random.default_rng(6)
    if case == "mixed":              # empty, short and cooperative rows (more than 32), rows over several warps and tiles, empty ends
        lens = rng.integers(0, 45, 40_000) * (rng.random(40_000) < 0.8)
        lens[rng.integers(0, 40_000, 40)] = rng.integers(200, 900, 40)
        lens[12_345], lens[:300], lens[-7:] = 30_000, 0, 0
        return lens
    if case == "ones":               # as many pieces to a region as there can be
        return np.ones(330_000, np.int64)
    if case == "one_row":            # no region but the last holds the end of a row
        return np.array([0, 700_000, 3])
    return np.concatenate([np.tile([31, 32, 33, 1, 2, 3, 4, 5], 6000), [2500]])      # "edges": both sides of a step of four and of the cooperative rows


def by_bundles(A, k, beta, dtype):
    plan = b200sp.b200sp_plan_create(A.m, A.n, A.nnz, to_dev(A.row_ptr))
    stats = b200sp.b200sp_plan_info(plan)
    b200sp.b200sp_plan_destroy(plan)
    return b200sp.b200sp_spmm_by_bundles(stats, k, beta, dtype)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("case", ["mixed", "ones", "one_row", "edges"])
def test_bundles_against_oracle(case, dtype):
    lens = lengths(case)
    n = 30_000
    A = gen.random_csr(len(lens), n, lens, seed=5, sort_cols=False)
    rng = np.random.default_rng(7)
    taken = 0
    b200sp.b200sp_set_option("spmm_flat", 1)
    try:
        for k in WIDTHS[dtype] if case in ("mixed", "edges") else WIDTHS[dtype][::3]:
            taken += by_bundles(A, k, 0.0, dtype) + by_bundles(A, k, 1.25, dtype)
            B = rng.standard_normal(n * k).astype(np.float32)
            Y0 = rng.standard_normal(A.m * k).astype(np.float32)
            Y, Y_ref, S = run_spmm(A, B, k, None, 1.0, 0.0, dtype)
            assert_within(Y, Y_ref, S, dtype, what="k=%d" % k)
            Y, Y_ref, S = run_spmm(A, B, k, Y0, -0.5, 1.25, dtype)
            y0f = Y0 if dtype == "f32" else gen.bf16_to_f32(gen.to_bf16(Y0))
            assert_within(Y, Y_ref, S, dtype, 1.0, np.abs(1.25 * y0f.astype(np.float64)).reshape(A.m, k), what="k=%d ab" % k)
    finally:
        b200sp.b200sp_set_option("spmm_flat", 2)
    assert taken >= 6, "the rule sends too few of these calls to the kernel"


@pytest.mark.parametrize("dtype,k", [("f32", 32), ("f32", 33), ("bf16", 64), ("bf16", 50)])
def test_infinities_stay_in_the_rows_that_hold_them(dtype, k):
    """Loads that stand in for missing nonzeros read the last row of B again: an infinity there must not turn into 0 * inf."""
    lens = np.tile([1, 2, 3, 5, 6, 7, 9, 40], 14_000)
    n = 20_000
    A = gen.random_csr(len(lens), n, lens, seed=9)
    B = np.random.default_rng(3).standard_normal((n, k)).astype(np.float32)
    B[::97] = np.inf
    B[5::97, ::3] = np.nan
    vals, Bs = store(A.vals, dtype), store(B.reshape(-1), dtype)
    d = [to_dev(a) for a in (A.row_ptr, A.col_idx, vals, Bs)]
    Y = empty_out(A.m * k, dtype)
    b200sp.b200sp_set_option("spmm_flat", 1)
    try:
        assert by_bundles(A, k, 0.0, dtype)
        b200sp.spmm_csr(A.m, n, A.nnz, k, d[0], d[1], d[2], d[3], Y, 1.0, 0.0, dtype)
    finally:
        b200sp.b200sp_set_option("spmm_flat", 2)
    got = to_host(Y, dtype)
    got = (got if dtype == "f32" else gen.bf16_to_f32(got)).reshape(A.m, k)
    ref, _ = oracle.spmm_csr(A.m, n, k, A.row_ptr, A.col_idx, vals, Bs, None, 1.0, 0.0, dtype)
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isposinf(got), np.isposinf(ref)) and np.array_equal(np.isneginf(got), np.isneginf(ref))


@pytest.mark.parametrize("dtype,k,length,rows", [("f32", 64, 7, 97_501), ("f32", 36, 5, 130_003), ("f32", 32, 9, 200_001), ("bf16", 72, 6, 111_500), ("bf16", 40, 11, 83_400)])
def test_equal_rows_of_odd_length(dtype, k, length, rows):
    """Just above the least number of items, in regions that cut rows at every place."""
    A = gen.uniform_rows(rows, 40_000, length, 2)
    assert by_bundles(A, k, 0.5, dtype)
    rng = np.random.default_rng(5)
    B, Y0 = rng.standard_normal(A.n * k).astype(np.float32), rng.standard_normal(A.m * k).astype(np.float32)
    Y, Y_ref, S = run_spmm(A, B, k, None, 1.0, 0.0, dtype)
    assert_within(Y, Y_ref, S, dtype)
    Y, Y_ref, S = run_spmm(A, B, k, Y0, 1.5, 0.5, dtype)
    y0f = Y0 if dtype == "f32" else gen.bf16_to_f32(gen.to_bf16(Y0))
    assert_within(Y, Y_ref, S, dtype, 1.5, np.abs(0.5 * y0f.astype(np.float64)).reshape(A.m, k))


@needs_plain_build
@pytest.mark.parametrize("pdl", [0, 1])
@pytest.mark.parametrize("dtype,k", [("bf16", 50), ("bf16", 33), ("f32", 33)])
def test_padded_calls_read_what_the_calls_just_before_them_wrote(dtype, k, pdl):
    """The copy of B, the walk and the fix-up wait for the stream's earlier work before anything is read or written: the values of A, B and the old values
    of Y all come from the calls just before, and a quarter of the rows are empty (Y of these is written first of all)."""
    rng = np.random.default_rng(8)
    m = 70_000
    lens = rng.integers(4, 19, m) * (rng.random(m) < 0.75)
    lens[5], lens[-1] = 3000, 0
    A = gen.random_csr(m, m, lens, seed=4)
    assert by_bundles(A, k, 0.5, dtype)
    one_each = gen.uniform_rows(A.nnz, A.nnz, 1, 3)               # a product that writes the values of A
    as_stored = torch.float32 if dtype == "f32" else torch.int16
    d = [to_dev(a) for a in (A.row_ptr, A.col_idx, one_each.row_ptr, one_each.col_idx, store(np.full(A.nnz, 0.25, np.float32), dtype))]
    x = [to_dev(store(rng.standard_normal(A.nnz).astype(np.float32), dtype)) for _ in range(2)]
    start = [to_dev(store(rng.standard_normal(m * k).astype(np.float32), dtype)) for _ in range(2)]
    plan = b200sp.b200sp_plan_create(A.m, A.n, A.nnz, d[0])
    plan_of_values = b200sp.b200sp_plan_create(A.nnz, A.nnz, A.nnz, d[2])

    def chain(wait):
        vals = torch.zeros(A.nnz, dtype=as_stored, device="cuda")
        P, Q = (t.clone() for t in start)
        torch.cuda.synchronize()
        for i in range(60):
            b200sp.b200sp_spmv(plan_of_values, d[3], d[4], x[i % 2], vals, 1.0, 0.0, dtype)
            wait()
            b200sp.b200sp_spmm(plan, k, d[1], vals, P, Q, 0.5, -0.5, dtype)
            wait()
            b200sp.b200sp_spmm(plan, k, d[1], vals, Q, P, 0.5, 0.25 if i % 3 else 0.0, dtype)
            wait()
        torch.cuda.synchronize()
        return P, Q

    b200sp.b200sp_set_option("pdl", 0)
    try:
        expected = chain(torch.cuda.synchronize)
        b200sp.b200sp_set_option("pdl", pdl)
        for _ in range(3):
            got = chain(lambda: None)
            assert all(torch.equal(a.view(torch.int16), b.view(torch.int16)) for a, b in zip(got, expected))
    finally:
        b200sp.b200sp_set_option("pdl", 1)
        b200sp.b200sp_plan_destroy(plan)
        b200sp.b200sp_plan_destroy(plan_of_values)
    values = expected[0] if dtype == "f32" else expected[0].view(torch.bfloat16)
    assert bool(torch.isfinite(values).all()) and float(values.float().abs().max()) > 0.0


@needs_plain_build
@pytest.mark.parametrize("dtype,k", [("bf16", 50), ("bf16", 63), ("bf16", 126), ("bf16", 127)])
def test_empty_rows_of_ragged_width_cost_little_more_than_their_bytes(dtype, k):
    """The same nonzeros with and without 250,000 empty rows behind them, whole regions of nothing else.  One column at a time by the lanes that hold a
    piece of B, these took longer than the products."""
    lens = np.random.default_rng(3).integers(2, 40, 100_000)
    n = len(lens)
    best = {}
    for empties in (0, 250_000):
        A = gen.random_csr(n + empties, n, np.concatenate([lens, np.zeros(empties, np.int64)]), seed=6, sort_cols=False)
        assert by_bundles(A, k, 0.0, dtype)
        d = [to_dev(a) for a in (A.row_ptr, A.col_idx, store(A.vals, dtype), store(np.ones(n * k, np.float32), dtype))]
        Y = empty_out(A.m * k, dtype)
        plan = b200sp.b200sp_plan_create(A.m, A.n, A.nnz, d[0])
        best[empties] = 1e9
        for _ in range(8):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            for _ in range(8):
                b200sp.b200sp_spmm(plan, k, d[1], d[2], d[3], Y, 1.0, 0.0, dtype)
            end.record()
            torch.cuda.synchronize()
            best[empties] = min(best[empties], start.elapsed_time(end) / 8)
        b200sp.b200sp_plan_destroy(plan)
    assert best[250_000] < 1.5 * best[0], "%.1f us, without the empty rows %.1f us" % (1e3 * best[250_000], 1e3 * best[0])


@pytest.mark.parametrize("dtype,full,holes", [("f32", ((33, 0.0), (63, 1.25), (16, 0.0)), ((36, 1.25), (64, 1.25), (100, 1.25), (128, 1.25), (33, 1.25), (63, 1.25), (17, 1.25), (9, 1.25))),
                                              ("bf16", ((72, 0.0), (120, 1.25), (128, 0.0), (127, 0.0), (65, 1.25), (126, 0.0), (50, 1.25)), ((72, 1.25), (128, 0.0), (128, 1.25), (33, 0.0), (127, 1.25), (50, 0.0), (34, 1.25)))])
def test_every_form_that_the_rules_take(dtype, full, holes):
    """Both matrices just large enough for the widest forms: rows of 1 to 40 and some longer than a region, without empty rows, and with 45 % of them, in long and short runs."""
    rng = np.random.default_rng(12)
    n = 30_000
    lens = rng.integers(1, 40, 52_000)
    lens[rng.integers(0, 52_000, 30)] = rng.integers(200, 1500, 30)
    with_holes = rng.integers(1, 40, 100_000) * (rng.random(100_000) < 0.75)
    with_holes[30_000:57_000] = 0
    for rows, calls in ((lens, full), (with_holes, holes)):
        A = gen.random_csr(len(rows), n, rows, seed=3, sort_cols=False)
        for k, beta in calls:
            assert by_bundles(A, k, beta, dtype), (k, beta)
            B, Y0 = rng.standard_normal(n * k).astype(np.float32), rng.standard_normal(A.m * k).astype(np.float32)
            Y, Y_ref, S = run_spmm(A, B, k, Y0 if beta else None, -0.5 if beta else 1.0, beta, dtype)
            y0f = Y0 if dtype == "f32" else gen.bf16_to_f32(gen.to_bf16(Y0))
            assert_within(Y, Y_ref, S, dtype, 1.0, np.abs(beta * y0f.astype(np.float64)).reshape(A.m, k), what="k=%d beta=%g" % (k, beta))


@pytest.mark.parametrize("k,beta,lens", [
    (32, 0.5, np.concatenate([np.repeat([0, 3], 5000), [30_000], np.full(200, 32), np.full(200, 33), np.zeros(3000, np.int64)])),     # regions of 24 items, the shortest
    (16, 0.0, np.concatenate([np.repeat([2, 5], 9000), [150_000], np.full(200, 33), np.full(400, 32), np.full(30, 87)])),             # just above the least number of items
    (64, 0.5, np.concatenate([np.repeat([0, 9], 60_000), [400_000], np.full(100, 1000)]))],
    ids=["regions_of_24", "least_items", "long_regions"])
def test_positive_data_stays_below_the_literal_fp32_bound(k, beta, lens):
    """All-positive data, where rounding errors do not cancel: a row over hundreds of tiles, pieces at the limit of the cooperative ones, full regions.  A row over T tiles adds at
    most 128 products in a chain, five levels of a tree, eight partial sums and a chain of T / 16 trees of 16: 600 tiles are 183 additions, 0.36 of the literal bound if all erred
    the same way."""
    n = 20_000
    A = gen.random_csr(len(lens), n, lens, seed=8, allow_dup=True)
    rng = np.random.default_rng(2)
    A.vals[:] = rng.random(A.nnz).astype(np.float32) + 0.01
    B = rng.random(n * k).astype(np.float32) + 0.01
    assert by_bundles(A, k, beta, "f32")
    Y, Y_ref, S = run_spmm(A, B, k, np.zeros(A.m * k, np.float32), 1.0, beta, "f32")
    assert assert_within(Y, Y_ref, S, "f32") < 0.5
