"""The plan pass (statistics written to pinned memory by its last block): sizes around its block and grid edges, passes one after
another (the accumulators must come back clean) and from several threads at once."""
import threading
import time

import numpy as np
import pytest
import torch

import paper_2603_07169_b200 as b200sp

pytestmark = pytest.mark.gpu
EDGES = [(0, 0), (1, 4), (5, 32), (33, 128), (129, 1024), (1025, 1 << 30)]


def expect(lens):
    rows = [int(((lens >= a) & (lens <= b)).sum()) for a, b in EDGES]
    nnz = [int(lens[(lens >= a) & (lens <= b)].sum()) for a, b in EDGES]
    return int(lens.min()), int(lens.max()), rows, nnz


def check(lens, stream=None):
    row_ptr = torch.from_numpy(np.concatenate([[0], lens.cumsum()]).astype(np.int32)).to("cuda:0")
    torch.cuda.synchronize()
    plan = b200sp.b200sp_plan_create(len(lens), 1 << 20, int(lens.sum()), row_ptr, stream)
    info = b200sp.b200sp_plan_info(plan)
    b200sp.b200sp_plan_destroy(plan)
    assert (info["min_row_len"], info["max_row_len"], info["bin_rows"], info["bin_nnz"]) == expect(lens)


def lengths(m, seed):
    rng = np.random.default_rng(seed)
    return rng.choice([0, 1, 4, 5, 32, 33, 128, 129, 700, 1024, 1025, 3000], m, p=[.2, .2, .1, .1, .1, .1, .05, .05, .04, .03, .02, .01]).astype(np.int64)


@pytest.mark.parametrize("m", [1, 31, 255, 256, 257, 1023, 1024, 1025, 4097, 1_300_000])
def test_statistics_match_numpy(m):
    for seed in range(3):
        check(lengths(m, seed))
    check(np.full(m, 7, np.int64))       # nothing left over from the passes before


@pytest.mark.parametrize("case", ["mixed", "longest_first", "longest_last", "several_long", "one_row", "all_empty_but_one", "rows_of_a_share", "rows_of_a_tile", "searched_four_rows_a_thread", "most_rows"])
def test_split_points_from_the_rows(case):
    """Tiles of SpMV and shares of SpMM cut where the pass says: sums of ones, which are the row lengths.  Rows that hold no split point, one,
    more than the sixteen that a lane writes alone and more than the 1024 that a warp does; the split points behind the last row.  Split points that
    are searched: one_row and rows_of_a_tile, which hold many to a row, and more rows (1.3 million) than the rows' form takes (most_rows is its largest)."""
    lens = {"mixed": lengths(3001, 5), "longest_first": np.concatenate([[150_000], np.full(999, 3)]), "longest_last": np.concatenate([np.full(999, 3), [150_000]]),
            "several_long": np.concatenate([np.full(900, 3), np.full(5, 140_000), np.full(1100, 2)]), "one_row": np.array([70_000]), "all_empty_but_one": np.concatenate([np.zeros(40_000), [5], np.zeros(9_000)]), "rows_of_a_share": np.full(500, 31),
            "rows_of_a_tile": np.full(64, 1023), "searched_four_rows_a_thread": np.random.default_rng(1).integers(0, 6, 1_300_000), "most_rows": np.random.default_rng(2).integers(0, 9, 1 << 17)}[case].astype(np.int64)
    m, nnz, k = len(lens), int(lens.sum()), 4
    row_ptr = torch.from_numpy(np.concatenate([[0], lens.cumsum()]).astype(np.int32)).to("cuda:0")
    col = torch.randint(0, 1000, (nnz,), dtype=torch.int32, device="cuda:0")
    ones, x = torch.ones(nnz, device="cuda:0"), torch.ones(1000 * k, device="cuda:0")
    want = torch.from_numpy(lens).to("cuda:0").float()
    b200sp.b200sp_set_option("spmv_kernel", 0)
    b200sp.b200sp_set_option("spmm_flat", 1)
    b200sp.b200sp_set_option("spmm_bstage", 0)
    try:
        for items in (0, 1024, 4096):
            b200sp.b200sp_set_option("merge_items", items)
            plan = b200sp.b200sp_plan_create(m, 1000, nnz, row_ptr)
            y, Y = torch.full((m,), float("nan"), device="cuda:0"), torch.full((m * k,), float("nan"), device="cuda:0")
            b200sp.b200sp_spmv(plan, col, ones, x, y, 1.0, 0.0, "f32")
            b200sp.b200sp_spmm(plan, k, col, ones, x, Y, 1.0, 0.0, "f32")
            b200sp.b200sp_plan_destroy(plan)
            assert torch.equal(y, want) and torch.equal(Y.view(m, k), want[:, None].expand(m, k))
    finally:
        for name, value in (("spmv_kernel", -1), ("spmm_flat", 2), ("spmm_bstage", 1), ("merge_items", 0)):
            b200sp.b200sp_set_option(name, value)


@pytest.mark.parametrize("rows,length", [(8, 200_000_000), (100, 21_000_000)])
def test_a_plan_of_few_rows_costs_no_more_than_one_of_many(rows, length):
    """100,000 to a million split points in a handful of rows: 200 us where the rows' own warp writes them all, 21 us where each is searched."""
    def create_us(row_ptr, m, nnz):
        times = []
        for _ in range(30):
            torch.cuda.synchronize()
            start = time.perf_counter()
            plan = b200sp.b200sp_plan_create(m, 1 << 20, nnz, row_ptr)
            times.append(time.perf_counter() - start)
            b200sp.b200sp_plan_destroy(plan)
        return 1e6 * sorted(times)[7]
    few = create_us((torch.arange(rows + 1, device="cuda:0") * length).int(), rows, rows * length)
    many = create_us((torch.arange((1 << 20) + 1, device="cuda:0") * 16).int(), 1 << 20, 1 << 24)
    assert few < 2.0 * many, "%.1f us, a million rows of 16 %.1f us" % (few, many)


def test_passes_from_several_threads():
    failures = []

    def work(i):
        try:
            s = torch.cuda.Stream()
            for j in range(20):
                check(lengths(1000 * i + 17 * j + 1, j), s)
        except BaseException as e:      # noqa: BLE001 - reported below
            failures.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures[0]


def test_a_capturing_stream_is_refused():
    """No pass is recorded and no accumulator lost (there are 64): the capture goes on, and later passes count from zero."""
    lens = lengths(5000, 1)
    row_ptr = torch.from_numpy(np.concatenate([[0], lens.cumsum()]).astype(np.int32)).to("cuda:0")
    x, graph = torch.zeros(8, device="cuda:0"), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(70):
            with pytest.raises(b200sp.B200spError) as e:
                b200sp.b200sp_plan_create(len(lens), 1 << 20, int(lens.sum()), row_ptr)
            assert e.value.status == 2      # B200SP_ERR_UNSUPPORTED
        x += 1
    graph.replay()
    torch.cuda.synchronize()
    assert x.sum().item() == 8
    for seed in range(70):
        check(lengths(3000, seed))
