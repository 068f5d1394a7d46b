"""SpMV of CSC matrices by products written in runs (csc_kernels.cuh): every tile and bucket size, ragged ends, rows and columns at the
limits of the path and beyond them (where the CSR kernels take over), and reproducible sums."""
import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2603_07169_b200 as b200sp
from gpu_util import assert_within, empty_out, needs_plain_build, store, to_dev, to_host

pytestmark = pytest.mark.gpu


def matrices():
    rng = np.random.default_rng(12)
    tail = np.zeros(4000, np.int64)
    tail[:50] = 30
    return {
        "one_entry": (np.array([0, 1, 0]), 5),
        "tile_less_one": (np.full(23, 89), 300),                  # 2047 nonzeros
        "tile_exact": (np.full(32, 64), 300),                     # 2048 nonzeros: one tile, one bucket
        "tile_plus_one": (np.full(3, 683), 900),                  # 2049 nonzeros
        "rows_at_the_limit": (np.array([1024] * 5 + [0, 1, 1024, 33, 32]), 2000),
        "row_over_the_limit": (np.array([1025] + [3] * 500), 2000),   # a bucket may still hold it
        "row_far_over": (np.array([5000] + [3] * 2000), 6000),    # CSR kernels
        "wide_tile": (np.full(3000, 2), 900_000),                 # a tile spans more than 65536 columns: CSR kernels
        "trailing_empty_rows": (tail, 100),
        "more_rows_than_a_bucket": (np.concatenate([tail, np.zeros(4000, np.int64), tail]), 100),
        # one bucket of 2048 nonzeros and as many rows as the products take (beta = 0 / beta != 0), and one more
        "bucket_rows_at_the_limit": (np.resize(np.repeat([32, 0], 64), 4224) * (np.arange(4224) < 128), 300),
        "bucket_rows_over_the_limit": (np.resize(np.repeat([32, 0], 64), 4225) * (np.arange(4225) < 128), 300),
        "bucket_rows_at_the_limit_of_beta": (np.resize(np.repeat([32, 0], 64), 2816) * (np.arange(2816) < 128), 300),
        "power_law": ((rng.pareto(1.5, 30_000) * 2).astype(np.int64).clip(0, 900), 20_000),
        "tile_4096": (rng.integers(0, 30, 100_000), 50_000),
        "tile_24576": (16, 328_000),                              # 5.2 M nonzeros (equal rows: drawn by the fast generator)
        "tile_28672": (16, 500_000),
        "tile_32768": (16, 560_000),
    }


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("case", sorted(matrices()))
def test_csc_products_against_oracle(case, dtype):
    lens, n = matrices()[case]
    A = gen.uniform_rows(n, n, lens, 3) if isinstance(lens, int) else gen.random_csr(len(lens), n, lens, seed=3, sort_cols=True)
    rng = np.random.default_rng(1)
    cp, ri, va = gen.csr_to_csc(A)
    v_s, x_s, y0_s = store(va, dtype), store(rng.standard_normal(n).astype(np.float32), dtype), store(rng.standard_normal(A.m).astype(np.float32), dtype)
    d = [to_dev(a) for a in (cp, ri, v_s, x_s)]
    y_ref, S = oracle.spmm_csc(A.m, n, 1, cp, ri, v_s, x_s, None, 1.0, 0.0, dtype)
    outs = []
    for _ in range(2):
        y = empty_out(A.m, dtype)
        b200sp.spmv_csc(A.m, n, A.nnz, d[0], d[1], d[2], d[3], y, 1.0, 0.0, dtype)
        outs.append(to_host(y, dtype))
        b200sp.b200sp_cache_drop(d[0])                            # the second pass plans again: the same sums in the same order
    assert_within(outs[0], y_ref[:, 0], S[:, 0], dtype, what=case)
    assert np.array_equal(outs[0], outs[1])
    y = to_dev(y0_s).clone()
    b200sp.spmv_csc(A.m, n, A.nnz, d[0], d[1], d[2], d[3], y, -0.5, 1.25, dtype)
    y_ref, S = oracle.spmm_csc(A.m, n, 1, cp, ri, v_s, x_s, y0_s, -0.5, 1.25, dtype)
    y0f = y0_s if dtype == "f32" else gen.bf16_to_f32(y0_s)
    assert_within(to_host(y, dtype), y_ref[:, 0], S[:, 0], dtype, 1.0, np.abs(1.25 * y0f.astype(np.float64)), what=case + " ab")
    b200sp.b200sp_cache_clear()


@pytest.mark.parametrize("per_row", [31, 33])
def test_csc_products_around_the_largest_bucket_size(per_row):
    """2^20 rows: nonzeros on both sides of 2^25, where buckets double; against 64-bit sums on the GPU."""
    m = 1 << 20
    g = torch.Generator("cuda").manual_seed(per_row)
    row = torch.arange(m, device="cuda").repeat_interleave(per_row)
    col = torch.randint(0, m, (m * per_row,), generator=g, device="cuda")
    key = (col * m + row).sort().values
    col, row = key // m, (key % m).int()
    cp = torch.searchsorted(col, torch.arange(m + 1, device="cuda")).int()
    vals = torch.randn(m * per_row, generator=g, device="cuda")
    x = torch.randn(m, generator=g, device="cuda")
    y = torch.full((m,), float("nan"), device="cuda")
    b200sp.spmv_csc(m, m, m * per_row, cp, row, vals, x, y, 1.0, 0.0, "f32")
    p = vals.double() * x.double()[col]
    ref = torch.zeros(m, dtype=torch.float64, device="cuda").index_add_(0, row.long(), p)
    S = torch.zeros(m, dtype=torch.float64, device="cuda").index_add_(0, row.long(), p.abs())
    assert float(((y.double() - ref).abs() / (1e-5 * S + 1e-30)).max()) <= 1.0
    b200sp.b200sp_cache_clear()


@pytest.mark.parametrize("beta", [0.0, 0.5])
def test_a_few_entries_in_many_rows(beta):
    """2000 entries in 2^22 rows are one bucket of products: one CTA would walk all rows (2.3 ms, 3.5 ms with beta != 0; 27 us by the CSR kernels)."""
    m, n, nnz = 1 << 22, 4096, 2000
    rng = np.random.default_rng(6)
    key = np.sort(rng.integers(0, n, nnz) * m + rng.integers(0, m, nnz))
    col, row = key // m, (key % m).astype(np.int32)
    cp = np.searchsorted(col, np.arange(n + 1)).astype(np.int32)
    va, x = rng.standard_normal(nnz).astype(np.float32), rng.standard_normal(n).astype(np.float32)
    d = [to_dev(a) for a in (cp, row, va, x)]
    y = torch.ones(m, device="cuda")
    call = lambda: b200sp.spmv_csc(m, n, nnz, d[0], d[1], d[2], d[3], y, 1.0, beta, "f32")  # noqa: E731
    call()
    p, at = va.astype(np.float64) * x[col], row.astype(np.int64)
    ref, S = beta + np.bincount(at, p, m), beta + np.bincount(at, np.abs(p), m)
    assert np.all(np.abs(y.cpu().numpy() - ref) <= 1e-5 * S + 1e-30)
    start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    best = 1e9
    for _ in range(5):
        start.record()
        call()
        end.record()
        torch.cuda.synchronize()
        best = min(best, start.elapsed_time(end))
    assert best < 0.5, "%.3f ms" % best
    b200sp.b200sp_cache_clear()


def test_dropping_a_csc_pattern_drops_the_plans_of_its_row_offsets():
    """Two patterns of the same sizes one after another under one address: the second must not meet anything of the first."""
    rng = np.random.default_rng(4)
    m, n = 4000, 3000
    lens1 = np.full(m, 8)
    lens2 = rng.integers(0, 17, m)
    lens2[:8] += 1500                                             # too long for the products: the CSR kernels and their plan
    lens1[0] += lens2.sum() - lens1.sum()
    ptr = None
    for lens in (lens1, lens2, lens1):
        A = gen.random_csr(m, n, lens, seed=2, sort_cols=True)
        cp, ri, va = gen.csr_to_csc(A)
        x = rng.standard_normal(n).astype(np.float32)
        if ptr is None:
            ptr, idx = to_dev(cp), to_dev(ri)
        ptr.copy_(torch.from_numpy(cp)), idx.copy_(torch.from_numpy(ri))
        y = empty_out(m, "f32")
        b200sp.spmv_csc(m, n, A.nnz, ptr, idx, to_dev(va), to_dev(x), y, 1.0, 0.0, "f32")
        y_ref, S = oracle.spmm_csc(m, n, 1, cp, ri, va, x, None, 1.0, 0.0, "f32")
        assert_within(to_host(y, "f32"), y_ref[:, 0], S[:, 0], "f32")
        b200sp.b200sp_cache_drop(ptr)
    b200sp.b200sp_cache_clear()


@needs_plain_build
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("first", ["spmv", "spmm"])
def test_the_other_operation_captured(first, dtype):
    """After one eager call, of SpMV or of SpMM, both can be captured.  What only the captured call needed goes with its graph."""
    rng = np.random.default_rng(5)
    m, n, k = 6000, 5000, 24
    A = gen.random_csr(m, n, rng.integers(2, 30, m), seed=4, sort_cols=True)
    cp, ri, va = gen.csr_to_csc(A)
    v_s, x_s, B_s = (store(a, dtype) for a in (va, rng.standard_normal(n).astype(np.float32), rng.standard_normal(n * k).astype(np.float32)))
    d = [to_dev(a) for a in (cp, ri, v_s, x_s, B_s)]
    calls = {"spmv": lambda y: b200sp.spmv_csc(m, n, A.nnz, d[0], d[1], d[2], d[3], y, 1.0, 0.0, dtype),
             "spmm": lambda y: b200sp.spmm_csc(m, n, A.nnz, k, d[0], d[1], d[2], d[4], y, 1.0, 0.0, dtype)}
    refs = {"spmv": oracle.spmm_csc(m, n, 1, cp, ri, v_s, x_s, None, 1.0, 0.0, dtype), "spmm": oracle.spmm_csc(m, n, k, cp, ri, v_s, B_s, None, 1.0, 0.0, dtype)}
    sizes = {"spmv": m, "spmm": m * k}

    def check(y, op, what):
        assert_within(to_host(y, dtype).reshape(refs[op][0].shape), *refs[op], dtype, what="%s %s" % (op, what))

    outs = {op: [empty_out(sizes[op], dtype) for _ in range(4)] for op in calls}
    for op, call in calls.items():                                # kernels loaded
        call(outs[op][3])
        check(outs[op][3], op, "eager")
    b200sp.b200sp_cache_clear()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for op, call in calls.items():                            # nothing is known of the pattern
            with pytest.raises(b200sp.B200spError) as e:
                call(outs[op][0])
            assert e.value.status == 2      # B200SP_ERR_UNSUPPORTED
    calls[first](outs[first][3])
    check(outs[first][3], first, "first")
    for op in (first, "spmm" if first == "spmv" else "spmv"):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            calls[op](outs[op][0])
        calls[op](outs[op][1])                                    # before the graph has run
        torch.cuda.synchronize()
        check(outs[op][1], op, "outside the graph")
        graph.replay()
        torch.cuda.synchronize()
        check(outs[op][0], op, "replayed")
        del graph
        calls[op](outs[op][2])
        torch.cuda.synchronize()
        assert torch.equal(outs[op][1], outs[op][2])
    b200sp.b200sp_cache_clear()


@pytest.mark.parametrize("n", [245_001, 455_000, 640_000], ids=["tile_4096_bucket_8192", "tile_8192_ragged", "tile_24576"])
def test_csc_products_of_the_sizes_between(n):
    """Tiles of 4096 with buckets of 8192, the last size in tiles of 8192 (7.28 M nonzeros) and one in tiles of 24576."""
    A = gen.uniform_rows(n, n, 16, 5)
    x = np.random.default_rng(2).standard_normal(n).astype(np.float32)
    cp, ri, va = gen.csr_to_csc(A)
    d = [to_dev(a) for a in (cp, ri, va, x)]
    y = empty_out(n, "f32")
    b200sp.spmv_csc(n, n, A.nnz, d[0], d[1], d[2], d[3], y, 1.0, 0.0, "f32")
    y_ref, S = oracle.spmm_csc(n, n, 1, cp, ri, va, x, None, 1.0, 0.0, "f32")
    assert_within(to_host(y, "f32"), y_ref[:, 0], S[:, 0], "f32")
    b200sp.b200sp_cache_clear()


def around_the_limits():
    """(number of nonzeros over that of SMs, nonzeros a row, tile, bucket): the last and the first size of each pair of tile and bucket."""
    return [(25 * 1024, 16, 4096, 8192), (8 * 4096 - 16, 16, 4096, 8192), (8 * 4096, 16, 8192, 8192), (6 * 8192 - 16, 16, 8192, 8192), (6 * 8192, 16, 24576, 8192), (6 * 8192 + 64, 16, 28672, 8192),
            (69_000, 16, 24576, 8192), (25 * 1024 - 16, 16, 4096, 4096), (27_000, 1, 4096, 4096)]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("per_sm,per_row,tile,bucket", around_the_limits())
def test_each_pair_of_tile_and_bucket_against_oracle(per_sm, per_row, tile, bucket, dtype):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m = per_sm * sms // per_row
    assert b200sp.b200sp_csc_sizes(m, m * per_row, sms) == (tile, bucket)
    A = gen.uniform_rows(m, m, per_row, 7)
    rng = np.random.default_rng(3)
    cp, ri, va = gen.csr_to_csc(A)
    v_s, x_s, y0_s = store(va, dtype), store(rng.standard_normal(m).astype(np.float32), dtype), store(rng.standard_normal(m).astype(np.float32), dtype)
    d = [to_dev(a) for a in (cp, ri, v_s, x_s)]
    outs = []
    for _ in range(2):
        y = to_dev(y0_s).clone()
        b200sp.spmv_csc(m, m, A.nnz, d[0], d[1], d[2], d[3], y, -0.5, 1.25, dtype)
        outs.append(to_host(y, dtype))
        b200sp.b200sp_cache_drop(d[0])                            # planned again: the same sums in the same order
    assert np.array_equal(outs[0], outs[1])
    y_ref, S = oracle.spmm_csc(m, m, 1, cp, ri, v_s, x_s, y0_s, -0.5, 1.25, dtype)
    y0f = y0_s if dtype == "f32" else gen.bf16_to_f32(y0_s)
    assert_within(outs[0], y_ref[:, 0], S[:, 0], dtype, 1.0, np.abs(1.25 * y0f.astype(np.float64)))
    b200sp.b200sp_cache_clear()


@needs_plain_build
@pytest.mark.parametrize("first,second", [(0.0, 0.5), (0.5, 0.0)])
def test_larger_buckets_do_not_keep_a_pattern_from_its_products(first, second):
    """4.4 M nonzeros in 200,000 rows and 20,000 empty ones in one run: whichever bucket holds the run has more rows than pay with beta != 0, so buckets of 4096 are
    tried as well, and taken with beta == 0.  And 4 M in 9 M rows, where the smaller buckets are taken as before there were larger ones."""
    rng = np.random.default_rng(9)
    n = 300_000
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for lens in (np.repeat([22, 0, 22], [150_000, 20_000, 50_000]), (rng.random(9_000_000) < 0.45).astype(np.int64)):
        A = gen.random_csr(len(lens), n, lens, seed=3, sort_cols=True)
        assert sms * 25 * 1024 <= A.nnz < sms * 8 * 4096
        cp, ri, va = gen.csr_to_csc(A)
        x, y0 = rng.standard_normal(n).astype(np.float32), rng.standard_normal(A.m).astype(np.float32)
        d = [to_dev(a) for a in (cp, ri, va, x)]
        for beta in (first, second):
            y = to_dev(y0).clone()
            b200sp.spmv_csc(A.m, n, A.nnz, d[0], d[1], d[2], d[3], y, 1.0, beta, "f32")
            y_ref, S = oracle.spmm_csc(A.m, n, 1, cp, ri, va, x, y0 if beta else None, 1.0, beta, "f32")
            assert_within(to_host(y, "f32"), y_ref[:, 0], S[:, 0], "f32", 1.0, np.abs(beta * y0.astype(np.float64)))
        b200sp.b200sp_cache_clear()


@pytest.mark.parametrize("m", [12_000_000])
def test_many_rows_and_few_nonzeros_keep_the_time_they_had(m):
    """4.8 M nonzeros in 12 M rows, beta != 0: 82 us by products in buckets of 4096; with larger buckets alone the CSR kernels took the call, 113 us."""
    nnz, n = 4_800_000, 1 << 20
    g = torch.Generator("cuda").manual_seed(3)
    key = (torch.randint(0, n, (nnz,), generator=g, device="cuda") * m + torch.randint(0, m, (nnz,), generator=g, device="cuda")).sort().values
    col, row = key // m, (key % m).int()
    cp = torch.searchsorted(col, torch.arange(n + 1, device="cuda")).int()
    vals, x, y = (torch.randn(k, generator=g, device="cuda") for k in (nnz, n, m))
    y0 = y.clone()
    call = lambda: b200sp.spmv_csc(m, n, nnz, cp, row, vals, x, y, 1.0, 0.5, "f32")  # noqa: E731
    call()
    ref = (0.5 * y0.double()).index_add_(0, row.long(), vals.double() * x.double()[col])
    S = (0.5 * y0.double()).abs().index_add_(0, row.long(), (vals.double() * x.double()[col]).abs())
    assert float(((y.double() - ref).abs() / (1e-5 * S + 1e-30)).max()) <= 1.0
    before = b200sp.b200sp_launch_count()
    call()
    assert b200sp.b200sp_checked_build() or b200sp.b200sp_launch_count() - before == 2      # the products and the sums
    b200sp.b200sp_cache_clear()
