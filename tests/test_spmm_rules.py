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
    assert b200sp.b200sp_spmm_by_shares(uneven, 64, 0.0, dtype) and b200sp.b200sp_spmm_by_shares(uneven, last, 0.0, dtype)
    for k in (last + 1, 2**31 // size, 2**31 // size + 1, 2**31 // size + 64, 2**31 - 8, 2**31 - 1):
        assert not b200sp.b200sp_spmm_by_shares(uneven, k, 0.0, dtype) and not b200sp.b200sp_spmm_by_shares(even, k, 0.0, dtype), k


# Row statistics as b200sp_plan_info reports them; which way is faster by 10 % or more was measured (log-normal rows of 12 with sigma 0.9, rows
# of 8 and one of 3000, R-MAT).
LOG_NORMAL_600K = info(600_000, 600_000, [661, 155_601, 408_047, 35_056, 635, 0], [0, 439_795, 4_924_230, 1_728_721, 107_298, 0], 509)
LOG_NORMAL_20K = info(20_000, 20_000, [24, 5203, 13_581, 1165, 27, 0], [0, 14_759, 163_217, 57_544, 4473, 0], 259)
ONE_LONG = info(600_000, 600_000, [0, 1671, 598_328, 0, 0, 1], [0, 6664, 4_793_260, 0, 0, 3000], 3000)
RMAT_20 = info(1 << 20, 1 << 20, [640_000, 200_000, 150_000, 45_000, 12_500, 1076], [0, 400_000, 1_700_000, 2_400_000, 2_300_000, 1_588_608], 20_000)


@pytest.mark.parametrize("beta", [0.0, 1.0])
@pytest.mark.parametrize("stats,f32,bf16", [(LOG_NORMAL_600K, {2, 3}, {2}), (ONE_LONG, {2, 3, 4, 8}, {2, 3, 8, 16}), (LOG_NORMAL_20K, set(), set()),
                                            (RMAT_20, set(), set())], ids=["log_normal_600k", "one_long", "log_normal_20k", "rmat"])
def test_uneven_rows_and_few_columns(stats, f32, bf16, beta):
    for dtype, by_rows in (("f32", f32), ("bf16", bf16)):
        for k in by_rows:
            assert not b200sp.b200sp_spmm_by_shares(stats, k, beta, dtype), (dtype, k)
        for k in (17, 20, 23, 40, 64) if by_rows else (2, 3, 4, 5, 8, 12, 16, 17, 24, 32, 64):
            assert b200sp.b200sp_spmm_by_shares(stats, k, beta, dtype), (dtype, k)


SMS, L2 = 148, 126 << 20


@pytest.mark.parametrize("m,n,k,shortest,longest,mean,wide", [
    # measured on both sides; rows all of one length that is a multiple of four, of any number and over a B of any size
    (1 << 19, 1 << 19, 256, 32, 32, 32, True), (8000, 8192, 64, 4, 4, 4, True), (1 << 20, 1 << 20, 128, 16, 16, 16, True),
    # other lengths: while a slice of B takes less than half of L2
    (350_000, 350_000, 64, 13, 13, 13, True), (550_000, 550_000, 64, 13, 13, 13, False),
    (464_000, 464_000, 64, 13, 13, 13, True), (465_000, 465_000, 64, 13, 13, 13, False),
    # short ones: not in less than a quarter of a wave, nor of less than five nonzeros in more than three waves
    (8000, 8192, 64, 5, 15, 10, False), (20_000, 20_000, 64, 5, 15, 10, True), (100_000, 100_000, 64, 2, 6, 4, True), (100_000, 100_000, 128, 2, 6, 4, False),
    (8000, 8192, 64, 25, 25, 25, True),
    (200_000, 200_000, 256, 1, 1, 1, True),
    # of 26 to 32: in one wave or in many
    (20_000, 20_000, 64, 20, 36, 28, True), (20_000, 20_000, 128, 20, 36, 28, False), (16_384, 16_384, 192, 30, 30, 30, False),
    (100_000, 100_000, 192, 20, 36, 28, True), (20_000, 20_000, 128, 12, 30, 21, True),
    # of more than 32: no odd ones of one length, others not in a second or third wave
    (20_000, 20_000, 256, 65, 65, 65, False), (200_000, 200_000, 64, 33, 33, 33, False), (16_000, 16_000, 128, 64, 64, 64, True),
    (26_000, 26_000, 128, 64, 64, 64, False), (54_000, 54_000, 128, 64, 64, 64, True), (20_000, 20_000, 192, 64, 128, 96, False),
    (100_000, 100_000, 192, 64, 128, 96, True), (200_000, 200_000, 128, 32, 32, 32, True), (26_000, 26_000, 128, 32, 32, 32, True),
    # widths that are no whole pieces, or too few of them
    (50_000, 50_000, 72, 16, 16, 16, False), (50_000, 50_000, 48, 16, 16, 16, False), (50_000, 50_000, 80, 16, 16, 16, True)])
def test_rows_of_b_in_pieces_of_32_bytes(m, n, k, shortest, longest, mean, wide):
    stats = dict(info(m, n, [0, 0, m, 0, 0, 0], [0, 0, m * mean, 0, 0, 0], longest), min_row_len=shortest)
    assert b200sp.b200sp_spmm_wide_pieces(stats, k, SMS, L2) == wide
    b200sp.b200sp_set_option("spmm_stage_a", 1)
    try:
        assert not b200sp.b200sp_spmm_wide_pieces(stats, k, SMS, L2)
    finally:
        b200sp.b200sp_set_option("spmm_stage_a", 2)


LARGE = info(150_001, 120_007, [175, 38_000, 103_000, 8_700, 126, 0], [0, 109_000, 1_250_000, 433_000, 20_000, 0], 400)
EMPTY = info(1 << 17, 1 << 17, [80_000, 25_000, 18_000, 5_600, 2_200, 272], [0, 50_000, 210_000, 300_000, 290_000, 198_576], 6000)


@pytest.mark.parametrize("stats,dtype,beta,taken,left", [
    (LARGE, "f32", 0.0, (4, 8, 12, 16, 20, 32, 17, 33, 63), (36, 64, 128, 132, 18, 34, 50, 65, 127)),
    (LARGE, "bf16", 1.0, (8, 32, 40, 64, 72, 128, 17, 33, 127, 18, 50, 126), (136, 256, 20, 36, 100, 129, 130)),
    (EMPTY, "f32", 1.0, (4, 32, 64, 100, 128), (132, 50)),
    (EMPTY, "bf16", 0.0, (8, 64, 128, 33, 50), (20, 136, 300)),
    (LOG_NORMAL_20K, "f32", 0.0, (4, 16), (20, 32, 64, 33)),
    (LOG_NORMAL_20K, "bf16", 1.0, (), (72, 128, 50)),
], ids=["f32", "bf16", "empty_f32", "empty_bf16", "small_f32", "small_bf16"])
def test_rows_side_by_side(stats, dtype, beta, taken, left):
    """Narrow rows of B, by pieces of 16 bytes and by how often a padded copy would be read; larger matrices only."""
    for k in taken:
        assert b200sp.b200sp_spmm_by_bundles(stats, k, beta, dtype), k
    for k in left:
        assert not b200sp.b200sp_spmm_by_bundles(stats, k, beta, dtype), k


@pytest.mark.parametrize("dtype,k,length,rows,taken", [
    ("f32", 64, 7, 97_500, True), ("f32", 64, 7, 97_499, False), ("f32", 64, 8, 1 << 20, False), ("f32", 64, 21, 1 << 20, False), ("f32", 68, 7, 1 << 20, False),
    ("f32", 32, 13, 357_143, True), ("f32", 32, 13, 357_142, False), ("f32", 32, 9, 200_000, True), ("bf16", 64, 10, 454_545, False), ("f32", 16, 13, 1 << 20, False), ("bf16", 64, 6, 142_858, True), ("bf16", 64, 6, 142_857, False),
    ("bf16", 128, 5, 130_000, True), ("bf16", 128, 4, 1 << 20, False), ("bf16", 136, 5, 1 << 20, False)])
def test_equal_rows_side_by_side(dtype, k, length, rows, taken):
    """Rows of one length of 5 to 13 that is no multiple of four, on both sides of each limit."""
    stats = dict(info(rows, rows, [0, 0, rows, 0, 0, 0], [0, 0, rows * length, 0, 0, 0], length), min_row_len=length)
    assert not b200sp.b200sp_spmm_by_shares(stats, k, 0.0, dtype)
    assert b200sp.b200sp_spmm_by_bundles(stats, k, 0.0, dtype) == taken


@pytest.mark.parametrize("switch,values", [("spmm_sliced", [0]), ("spmm_flat", [0]), ("spmm_stage_a", [0, 1]), ("spmm_ranges", [0, 2, 3, 4, 8])])
@pytest.mark.parametrize("dtype,k,rows", [("bf16", 64, 1 << 20), ("f32", 64, 1 << 20), ("bf16", 128, 130_000)])
def test_equal_rows_stay_by_rows_where_a_switch_asks_for_it(dtype, k, rows, switch, values):
    stats = dict(info(rows, rows, [0, 0, rows, 0, 0, 0], [0, 0, rows * 7, 0, 0, 0], 7), min_row_len=7)
    default = b200sp.b200sp_get_option(switch)
    assert b200sp.b200sp_spmm_by_bundles(stats, k, 0.0, dtype)
    try:
        for value in values:
            b200sp.b200sp_set_option(switch, value)
            assert not b200sp.b200sp_spmm_by_bundles(stats, k, 0.0, dtype), value
    finally:
        b200sp.b200sp_set_option(switch, default)
    assert b200sp.b200sp_spmm_by_bundles(stats, k, 0.0, dtype)


def uneven(m, n, per_row, empty=0.0):
    """per_row nonzeros a row on average, `empty` of the rows without any, and eleven long rows."""
    none, nnz = int(m * empty), m * per_row
    return info(m, n, [none, 0, m - none - 11, 0, 10, 1], [0, 0, nnz - 10_000, 0, 5000, 5000], 5000)


@pytest.mark.parametrize("stats,dtype,k,beta,taken", [
    # measured by shares and side by side; BF16 with odd k above 32: short rows are not
    (uneven(50_000, 100_000, 14), "bf16", 33, 0.0, True), (uneven(200_000, 100_000, 4), "bf16", 63, 0.0, False), (uneven(800_000, 800_000, 9), "bf16", 127, 0.0, True),
    (uneven(50_000, 50_000, 6), "bf16", 127, 1.0, False), (uneven(25_000, 12_500, 14), "bf16", 95, 0.0, True),
    # many empty rows, old values of Y read: the copy may be large but for narrow rows
    (uneven(1 << 18, 1 << 18, 8, 0.6), "bf16", 50, 1.0, True), (uneven(1 << 21, 1 << 21, 8, 0.6), "f32", 63, 1.0, True), (uneven(1 << 18, 1 << 18, 8, 0.6), "f32", 17, 1.0, True),
    (uneven(1 << 18, 1 << 18, 8, 0.6), "bf16", 3, 1.0, True), (uneven(1 << 19, 1 << 19, 8, 0.6), "bf16", 3, 1.0, False), (uneven(1 << 18, 1 << 18, 6, 0.6), "bf16", 50, 1.0, False),
    # many empty rows that are only written: BF16, in two waves or more, from copies that stay in L2
    (uneven(1 << 18, 1 << 18, 8, 0.6), "bf16", 50, 0.0, True), (uneven(1 << 19, 1 << 19, 8, 0.6), "bf16", 50, 0.0, False), (uneven(1 << 17, 1 << 17, 8, 0.6), "bf16", 127, 0.0, False),
    (uneven(1 << 18, 1 << 18, 8, 0.6), "bf16", 127, 0.0, True), (uneven(1 << 19, 1 << 19, 8, 0.6), "bf16", 33, 0.0, True), (uneven(1 << 18, 1 << 18, 8, 0.6), "bf16", 17, 0.0, False),
    (uneven(1 << 18, 1 << 18, 8, 0.6), "f32", 63, 0.0, False), (uneven(1 << 18, 1 << 18, 8, 0.6), "f32", 9, 0.0, True), (uneven(1 << 17, 1 << 17, 8, 0.6), "bf16", 9, 0.0, False),
    # odd k of 17 to 31 without old values: small copies, read often
    (uneven(100_000, 100_000, 24), "f32", 17, 0.0, True), (uneven(100_000, 100_000, 14), "f32", 17, 0.0, False), (uneven(100_000, 100_000, 14), "f32", 17, 1.0, True),
    (uneven(150_000, 150_000, 24), "bf16", 31, 0.0, False),
    # the rest: how often a row of the copy is read, and whether it stays in L2
    (uneven(200_000, 200_000, 9), "bf16", 50, 0.0, False), (uneven(200_000, 100_000, 9), "bf16", 50, 0.0, True), (uneven(200_000, 200_000, 9), "bf16", 50, 1.0, True),
    (uneven(400_000, 400_000, 14), "f32", 63, 0.0, True), (uneven(400_000, 400_000, 14), "f32", 63, 1.0, False), (uneven(400_000, 400_000, 14), "bf16", 50, 0.0, False),
    (uneven(400_000, 400_000, 16), "bf16", 50, 0.0, True), (uneven(1_000_000, 1_000_000, 10), "f32", 5, 0.0, False), (uneven(150_000, 150_000, 11), "f32", 5, 0.0, True),
    (uneven(45_000, 45_000, 11), "f32", 5, 0.0, False), (uneven(1_000_000, 1_000_000, 10), "bf16", 2, 0.0, False), (uneven(45_000, 45_000, 11), "bf16", 10, 0.0, False),
    (uneven(60_000, 60_000, 11), "bf16", 10, 0.0, True)])
def test_a_padded_copy_of_b_only_where_it_pays(stats, dtype, k, beta, taken):
    assert b200sp.b200sp_spmm_by_shares(stats, k, beta, dtype)
    assert b200sp.b200sp_spmm_by_bundles(stats, k, beta, dtype) == taken


@pytest.mark.parametrize("dtype,k,length,items,beta,taken", [
    # measured on both sides: by what the length leaves over, the number of items and the kernel by rows that would take the call
    ("f32", 36, 13, 800_000, 0.0, False), ("f32", 36, 6, 800_000, 0.0, False), ("f32", 36, 10, 2_100_000, 1.0, False), ("f32", 64, 10, 800_000, 0.0, False),
    ("f32", 64, 9, 1_500_000, 0.0, True), ("f32", 48, 13, 3_200_000, 0.0, True), ("f32", 32, 11, 2_100_000, 0.0, False), ("f32", 20, 7, 2_100_000, 0.0, True),
    ("bf16", 64, 13, 2_100_000, 1.0, False), ("bf16", 64, 9, 1_050_000, 0.0, False), ("bf16", 64, 9, 3_200_000, 0.0, True), ("bf16", 64, 10, 5_100_000, 1.0, False),
    ("bf16", 64, 11, 2_100_000, 1.0, False), ("bf16", 40, 9, 1_050_000, 1.0, True), ("bf16", 40, 13, 1_050_000, 1.0, False), ("bf16", 72, 13, 800_000, 1.0, True),
    ("bf16", 128, 13, 5_100_000, 1.0, False), ("bf16", 128, 13, 5_100_000, 0.0, True), ("bf16", 128, 10, 800_000, 0.0, False), ("bf16", 96, 6, 800_000, 1.0, False),
    ("bf16", 128, 7, 800_000, 1.0, True)])
def test_equal_rows_side_by_side_only_where_they_are_faster(dtype, k, length, items, beta, taken):
    rows = -(-items // (length + 1))
    stats = dict(info(rows, rows, [0, 0, rows, 0, 0, 0], [0, 0, rows * length, 0, 0, 0], length), min_row_len=length)
    assert b200sp.b200sp_spmm_by_bundles(stats, k, beta, dtype) == taken


@pytest.mark.parametrize("stats,dtype,k,beta,taken", [
    # measured on both sides: BF16, nine to sixteen pieces of a row of B
    (uneven(124_000, 62_000, 4), "bf16", 128, 0.0, False), (uneven(100_000, 100_000, 8), "bf16", 128, 0.0, True), (uneven(320_000, 160_000, 4), "bf16", 72, 0.0, False),
    (uneven(320_000, 160_000, 4), "bf16", 72, 1.0, True), (uneven(1_000_000, 500_000, 8), "bf16", 72, 1.0, False), (uneven(60_000, 120_000, 9, 0.12), "bf16", 128, 0.0, False),
    (uneven(200_000, 240_000, 9, 0.12), "bf16", 128, 0.0, True), (uneven(600_000, 720_000, 9, 0.12), "bf16", 128, 0.0, False), (uneven(1 << 20, 1 << 20, 8, 0.6), "bf16", 128, 0.0, True),
    # old values of Y and empty rows
    (uneven(7000, 9000, 14, 0.12), "f32", 32, 1.0, False), (uneven(20_000, 24_000, 9, 0.12), "f32", 32, 1.0, True), (uneven(1 << 13, 1 << 13, 8, 0.6), "f32", 32, 1.0, True),
    (uneven(20_000, 24_000, 14, 0.12), "f32", 48, 1.0, False), (uneven(60_000, 72_000, 9, 0.12), "f32", 64, 1.0, True), (uneven(1 << 14, 1 << 14, 8, 0.6), "f32", 64, 1.0, True),
    (uneven(1 << 13, 1 << 13, 8, 0.6), "bf16", 128, 1.0, False), (uneven(1 << 15, 1 << 15, 8, 0.6), "bf16", 128, 1.0, True), (uneven(60_000, 72_000, 9, 0.12), "f32", 128, 1.0, False), (uneven(600_000, 1_200_000, 14, 0.12), "bf16", 72, 1.0, False),
    (uneven(1 << 15, 1 << 15, 8, 0.6), "f32", 128, 1.0, True), (uneven(1 << 14, 1 << 14, 8, 0.6), "f32", 128, 1.0, False)])
def test_wide_rows_of_b_side_by_side_only_where_they_are_faster(stats, dtype, k, beta, taken):
    assert b200sp.b200sp_spmm_by_shares(stats, k, beta, dtype)
    assert b200sp.b200sp_spmm_by_bundles(stats, k, beta, dtype) == taken
