"""Rows all of one length with scattered columns (spmv_equal_rows_kernel): one launch, every group size, a last warp that is not full."""
import numpy as np
import pytest
import torch

import gen
import paper_2603_07169_b200 as b200sp
from gpu_util import assert_within, empty_out, run_spmv, store, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("length", [3, 5, 15, 17, 31, 33, 63])
def test_equal_rows_against_oracle(length, dtype):
    rng = np.random.default_rng(length)
    for extra in (1, 7, 32, 127):
        m = ((1 << 20) // length // 128 + 1) * 128 + extra          # just above the small-problem kernel's range
        A = gen.random_csr(m, 300_000, np.full(m, length), seed=extra, sort_cols=False)
        x, y0 = rng.standard_normal(A.n).astype(np.float32), rng.standard_normal(m).astype(np.float32)
        y, y_ref, S = run_spmv(A, x, None, 1.0, 0.0, dtype)
        assert_within(y, y_ref, S, dtype, what="L=%d m=%d" % (length, m))
        y, y_ref, S = run_spmv(A, x, y0, -0.5, 1.25, dtype)
        y0f = y0 if dtype == "f32" else gen.bf16_to_f32(gen.to_bf16(y0))
        assert_within(y, y_ref, S, dtype, 1.0, np.abs(1.25 * y0f.astype(np.float64)), what="L=%d m=%d ab" % (length, m))


@pytest.mark.parametrize("length,launches", [(63, 1), (65, 2)])
def test_up_to_64_by_one_launch(length, launches):
    m = 30_000
    A = gen.random_csr(m, 300_000, np.full(m, length), seed=1, sort_cols=False)
    d = [to_dev(a) for a in (A.row_ptr, A.col_idx, store(A.vals, "f32"), store(np.ones(A.n, np.float32), "f32"))]
    y = empty_out(m, "f32")
    counts = []
    for _ in range(2):
        n0 = b200sp.b200sp_launch_count()
        b200sp.spmv_csr(m, A.n, A.nnz, d[0], d[1], d[2], d[3], y, 1.0, 0.0, "f32")
        torch.cuda.synchronize()
        counts.append(b200sp.b200sp_launch_count() - n0)
    b200sp.b200sp_cache_clear()
    assert b200sp.b200sp_checked_build() or counts[1] == launches
