"""The sizes of CSC SpMV by products, on the host (no GPU needed)."""
import pytest

import paper_2603_07169_b200 as b200sp

SMS = 148


@pytest.mark.parametrize("m,nnz,tile,bucket", [
    (1000, 1, 2048, 2048), (100_000, SMS * 4 * 2048 - 1, 2048, 2048), (100_000, SMS * 4 * 2048, 4096, 4096),
    # buckets of 8192 where rows have two nonzeros on average, or one from 4.2 M on
    (200_000, SMS * 25 * 1024 - 1, 4096, 4096), (200_000, SMS * 25 * 1024, 4096, 8192), (1_950_000, 3_900_000, 4096, 8192), (1_950_001, 3_900_000, 4096, 4096),
    (4_300_000, 4_300_000, 4096, 8192), (4_300_001, 4_300_000, 4096, 4096), (1 << 24, 4_800_000, 4096, 4096),
    # above, tiles of 8192 whatever the rows, and one large tile per SM and round from 7.3 M on
    (1 << 24, SMS * 8 * 4096, 8192, 8192), (200_000, SMS * 6 * 8192 - 1, 8192, 8192), (200_000, SMS * 6 * 8192, 24576, 8192), (455_000, 7_280_000, 28672, 8192), (640_000, 10_240_000, 24576, 8192),
    (1 << 20, 1 << 24, 28672, 8192), (1 << 20, 1 << 25, 32768, 8192), (1 << 20, (1 << 25) + 1, 32768, 16384)])
def test_tiles_and_buckets(m, nnz, tile, bucket):
    assert b200sp.b200sp_csc_sizes(m, nnz, SMS) == (tile, bucket)


def test_sizes_that_make_no_sense_are_refused():
    for m, nnz, sms in ((-1, 0, SMS), (0, -1, SMS), (0, 0, 0)):
        with pytest.raises(b200sp.B200spError):
            b200sp.b200sp_csc_sizes(m, nnz, sms)
