"""The native marshalling of the binding (csrc/marshal.cpp): what it does not take as it stands comes back as -1 and is refused, or handled,
by the Python path, exactly as before; what it takes reaches the library."""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

import gen
import oracle
import paper_2603_07169_b200 as b200sp
from paper_2603_07169_b200 import binding


def native():
    if binding._product is None:
        binding._load_native()
    return binding._product


def call(**change):
    a = dict(layout=0, m=4, n=4, nnz=4, k=0, a=None, b=None, vals=None, x=None, y=None, alpha=1.0, beta=0.0, dtype="f32", stream=1)
    a.update(change)
    return native()(binding._address["spmv_csr"], *a.values())


def test_unusual_arguments_are_left_to_python():
    assert call(m=0, n=5, nnz=0) == 0                                 # an empty problem is a no-op
    assert call(m=-1, nnz=0) == 1                                     # the library's own status
    for change in (dict(m=4.0), dict(m="4"), dict(alpha="1"), dict(dtype="f16"), dict(dtype=7), dict(dtype=None), dict(k=-1),
                   dict(m=1 << 80), dict(stream="x"), dict(x=np.zeros(4, np.float32)), dict(x=torch.zeros(4)), dict(a=[0, 1])):
        assert call(**change) == -1, change
    assert native()(1, 2, 3) == -1


def test_sizes_whose_products_64_bits_do_not_hold():
    """A wrapped product would let a short operand pass.  Left to Python, which counts exactly; the library refuses such sizes as well."""
    mm = binding._address if native() else None
    for m, n, nnz, k in ((4, 4, 4, 1 << 62), (4, 1 << 32, 4, 1 << 32), (1 << 32, 4, 4, 1 << 32), ((1 << 63) - 1, 4, 4, 1)):
        assert native()(mm["spmm_csr"], 0, m, n, nnz, k, None, None, None, None, None, 1.0, 0.0, "f32", 1) == -1
    assert native()(mm["spmv_csc"], 2, 4, (1 << 63) - 1, 4, 0, None, None, None, None, None, 1.0, 0.0, "f32", 1) == -1
    for m, n, width, k in ((1 << 30, 4, 1 << 34, 0), (1 << 30, 4, 1 << 34, 2), (4, 1 << 40, 4, 1 << 40)):
        assert binding._ell_product(mm["spmm_ell" if k else "spmv_ell"], m, n, width, k, None, None, None, None, 1.0, 0.0, "f32", 1) == -1
    assert binding._plan_create(mm["b200sp_plan_create"], (1 << 63) - 1, 4, 4, None, 1) == -1
    L, y = b200sp.lib(), np.zeros(16, np.float32)
    for width in (1 << 34, 1 << 62):                                  # m * width = 0 modulo 2^64
        assert L.spmv_ell(1 << 30, 4, width, None, None, None, y.ctypes.data, 1.0, 0.0, 0, None) == 1
        assert L.spmm_ell(1 << 30, 4, width, 2, None, None, None, y.ctypes.data, 1.0, 0.0, 0, None) == 1


def test_an_exception_out_of_the_call_becomes_a_status(tmp_path):
    """In place of the library: functions that run out of host memory.  The interpreter lock is held again afterwards."""
    (tmp_path / "throws.cpp").write_text("#include <new>\nextern \"C\" int f() { throw std::bad_alloc(); }\n"
                                         "extern \"C\" int info(const void*, void* out) { for (int i = 0; i < 144; ++i) ((char*)out)[i] = 0; return 0; }\n")
    lib = str(tmp_path / "throws.so")
    subprocess.check_call(["g++", "-shared", "-fPIC", "-o", lib, str(tmp_path / "throws.cpp")])
    L = ctypes.CDLL(lib)
    f, info = (ctypes.cast(getattr(L, n), ctypes.c_void_p).value for n in ("f", "info"))
    nothing = [None] * 5
    native()
    for _ in range(3):
        assert binding._product(f, 0, 0, 0, 0, 0, *nothing, 1.0, 0.0, "f32", 1) == 4      # B200SP_ERR_ALLOC
        assert binding._ell_product(f, 0, 0, 0, 0, *nothing[1:], 1.0, 0.0, "f32", 1) == 4
        assert binding._plan_product(info, f, 16, 0, *nothing[1:], 1.0, 0.0, "f32", 1) == 4
        assert binding._plan_create(f, 0, 0, 0, None, 1) == -2 - 4
        assert sum(range(1000)) == 499500


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_every_entry_point_through_it(dtype):
    from gpu_util import assert_within, empty_out, store, to_dev, to_host
    rng = np.random.default_rng(1)
    m, n, k = 300, 200, 24
    A = gen.random_csr(m, n, rng.integers(0, 9, m), 3, sort_cols=True)
    v, x, B = store(A.vals, dtype), store(rng.standard_normal(n).astype(np.float32), dtype), store(rng.standard_normal(n * k).astype(np.float32), dtype)
    d = [to_dev(a) for a in (A.row_ptr, A.col_idx, v, x, B)]
    rows, cols, _ = gen.csr_to_coo(A)
    cp, ri, cv = gen.csr_to_csc(A)
    w, ec, ev = gen.csr_to_ell(A)
    coo, csc, ell = [to_dev(a) for a in (rows, cols, v)], [to_dev(a) for a in (cp, ri, store(cv, dtype))], [to_dev(a) for a in (ec, store(ev, dtype))]
    plan = b200sp.b200sp_plan_create(m, n, A.nnz, d[0])
    stream = torch.cuda.Stream()
    y_ref, S = oracle.spmv_csr(m, n, A.row_ptr, A.col_idx, v, x, None, 1.0, 0.0, dtype)
    Y_ref, S2 = oracle.spmm_csr(m, n, k, A.row_ptr, A.col_idx, v, B, None, 1.0, 0.0, dtype)
    spmv = [lambda y, s: b200sp.spmv_csr(m, n, A.nnz, d[0], d[1], d[2], d[3], y, 1.0, 0.0, dtype, s),
            lambda y, s: b200sp.spmv_csr_noalloc(m, n, A.nnz, d[0], d[1], d[2], d[3], y, 1.0, 0.0, dtype, stream=s),
            lambda y, s: b200sp.spmv_coo(m, n, A.nnz, coo[0], coo[1], coo[2], d[3], y, 1, 0, dtype, s),
            lambda y, s: b200sp.spmv_csc(m, n, A.nnz, csc[0], csc[1], csc[2], d[3], y, 1.0, 0.0, dtype, s),
            lambda y, s: b200sp.spmv_ell(m, n, w, ell[0], ell[1], d[3], y, 1.0, 0.0, dtype, s),
            lambda y, s: b200sp.b200sp_spmv(plan, d[1], d[2], d[3], y, 1.0, 0.0, dtype, s),
            lambda y, s: b200sp.b200sp_spmv_naive(m, n, A.nnz, d[0], d[1], d[2], d[3], y, 1.0, 0.0, {"f32": 0, "bf16": 1}[dtype], s),
            lambda y, s: b200sp.spmv_csr(np.int64(m), n, A.nnz, d[0], d[1], d[2], d[3], y, np.float32(1.0), 0.0, dtype, s)]    # the Python path
    spmm = [lambda y, s: b200sp.spmm_csr(m, n, A.nnz, k, d[0], d[1], d[2], d[4], y, 1.0, 0.0, dtype, s),
            lambda y, s: b200sp.spmm_coo(m, n, A.nnz, k, coo[0], coo[1], coo[2], d[4], y, 1.0, 0.0, dtype, s),
            lambda y, s: b200sp.spmm_csc(m, n, A.nnz, k, csc[0], csc[1], csc[2], d[4], y, 1.0, 0.0, dtype, s),
            lambda y, s: b200sp.spmm_ell(m, n, w, k, ell[0], ell[1], d[4], y, 1.0, 0.0, dtype, s),
            lambda y, s: b200sp.b200sp_spmm(plan, k, d[1], d[2], d[4], y, 1.0, 0.0, dtype, s),
            lambda y, s: b200sp.b200sp_spmm_naive(m, n, A.nnz, k, d[0], d[1], d[2], d[4], y, 1.0, 0.0, dtype, s)]
    for calls, count, ref, bound in ((spmv, m, y_ref, S), (spmm, m * k, Y_ref, S2)):
        for i, f in enumerate(calls):
            for s in (None, stream, stream.cuda_stream):
                torch.cuda.synchronize()
                y = empty_out(count, dtype)
                torch.cuda.synchronize()
                f(y, s)
                torch.cuda.synchronize()
                assert_within(to_host(y, dtype).reshape(ref.shape), ref, bound, dtype, what="call %d" % i)
            for bad in (empty_out(count - 1, dtype), empty_out(count, "bf16" if dtype == "f32" else "f32"), empty_out(2 * count, dtype)[::2], torch.zeros(count)):
                with pytest.raises(b200sp.B200spError) as e:
                    f(bad, None)
                assert e.value.status == 1
    b200sp.b200sp_plan_destroy(plan)
    b200sp.b200sp_cache_clear()
