// Native argument marshalling of the Python binding: the checks that binding.py makes on every operand of a device call (a
// contiguous CUDA tensor on the current device with the right element size and enough elements), the current stream, and the
// call itself, without the interpreter in between.  In Python the same checks and the foreign call cost 9 us per call, as much as
// twice the kernels of small problems.
//
// Every function returns the library's status, or -1 for anything it does not take as it stands (a wrong tensor, an unusual
// argument type): the binding then goes through its Python path, which raises the precise error or handles the case.
#include <Python.h>
#include <ATen/core/Tensor.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <new>
#include <stdexcept>

#include "../../include/b200sp.h"

namespace {

struct Reader {
  bool ok = true;
  int device = -1;      // current device, looked up for the first tensor

  int current() {
    if (device < 0) device = c10::cuda::current_device();
    return device;
  }
  int64_t size(PyObject* o) {
    if (!PyLong_CheckExact(o)) { ok = false; return 0; }
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) { PyErr_Clear(); ok = false; }
    return v;
  }
  float scalar(PyObject* o) {
    if (PyFloat_CheckExact(o)) return (float)PyFloat_AS_DOUBLE(o);
    if (PyLong_CheckExact(o)) {
      const double v = PyLong_AsDouble(o);
      if (v == -1.0 && PyErr_Occurred()) { PyErr_Clear(); ok = false; }
      return (float)v;
    }
    ok = false;
    return 0.0f;
  }
  int dtype(PyObject* o) {
    if (PyUnicode_CheckExact(o)) {
      if (PyUnicode_CompareWithASCIIString(o, "f32") == 0) return B200SP_F32;
      if (PyUnicode_CompareWithASCIIString(o, "bf16") == 0) return B200SP_BF16;
    } else if (PyLong_CheckExact(o)) {
      const long v = PyLong_AsLong(o);
      if (v == B200SP_F32 || v == B200SP_BF16) return (int)v;
      PyErr_Clear();
    }
    ok = false;
    return 0;
  }
  // The product of two sizes; one that 64 bits do not hold is left to Python, whose integers do.
  int64_t times(int64_t a, int64_t b) {
    int64_t v = 0;
    if (__builtin_mul_overflow(a, b, &v)) ok = false;
    return v;
  }
  int64_t plus1(int64_t a) {
    if (a == INT64_MAX) ok = false;
    return ok ? a + 1 : a;
  }
  // Address of a device operand of at least `elems` elements of `esize` bytes; None stays NULL.
  void* operand(PyObject* o, int64_t elems, int64_t esize) {
    if (!ok || o == Py_None) return nullptr;
    if (!THPVariable_Check(o)) { ok = false; return nullptr; }
    const at::Tensor& t = THPVariable_Unpack(o);
    ok = t.is_cuda() && t.get_device() == current() && (int64_t)t.element_size() == esize && t.numel() >= elems && t.is_contiguous();
    return ok ? t.data_ptr() : nullptr;
  }
  void* stream(PyObject* o) {
    if (!ok) return nullptr;
    if (o == Py_None) return c10::cuda::getCurrentCUDAStream(current()).stream();
    PyObject* handle = nullptr;
    if (PyLong_CheckExact(o)) { handle = o; Py_INCREF(o); }
    else handle = PyObject_GetAttrString(o, "cuda_stream");
    void* s = nullptr;
    if (handle) { s = PyLong_AsVoidPtr(handle); Py_DECREF(handle); }
    if (PyErr_Occurred()) { PyErr_Clear(); ok = false; }
    return s;
  }
  void* address(PyObject* o) {
    void* p = PyLong_CheckExact(o) ? PyLong_AsVoidPtr(o) : nullptr;
    if (PyErr_Occurred()) PyErr_Clear();
    if (!p) ok = false;
    return p;
  }
};

template <typename Body>
PyObject* guarded(Body body) {
  int status = -1;
  try {
    status = body();
  } catch (...) {      // e.g. no device: the Python path reports it
    status = -1;
  }
  return PyLong_FromLong(status);
}

// A call of the library without the interpreter lock.  An exception that leaves it (out of host memory) becomes a status, and the lock is
// held again whichever way the call ends.
template <typename Call>
int unlocked(Call call) {
  struct Released {
    PyThreadState* state = PyEval_SaveThread();
    ~Released() { PyEval_RestoreThread(state); }
  } released;
  try {
    return call();
  } catch (const std::bad_alloc&) {
    return B200SP_ERR_ALLOC;
  } catch (const std::exception&) {
    return B200SP_ERR_CUDA;
  }
}

int64_t atleast0(int64_t v) { return v > 0 ? v : 0; }

// (fn, layout, m, n, nnz, k, a, b, vals, in, out, alpha, beta, dtype, stream); k == 0: SpMV.  layout 0: CSR (a = row_ptr, b = col_idx),
// 1: COO (a = row_idx, b = col_idx), 2: CSC (a = col_ptr, b = row_idx).
PyObject* product(PyObject*, PyObject* const* v, Py_ssize_t argc) {
  return guarded([&]() -> int {
    if (argc != 15) return -1;
    Reader r;
    void* const fn = r.address(v[0]);
    const int64_t layout = r.size(v[1]), m = r.size(v[2]), n = r.size(v[3]), nnz = r.size(v[4]), k = r.size(v[5]);
    const float alpha = r.scalar(v[11]), beta = r.scalar(v[12]);
    const int dtype = r.dtype(v[13]);
    if (!r.ok || k < 0) return -1;
    const int64_t e = dtype == B200SP_F32 ? 4 : 2, kk = k > 1 ? k : 1;
    const int64_t na = layout == 0 ? (m > 0 ? r.plus1(m) : 0) : layout == 1 ? nnz : r.plus1(n);
    const int32_t* a = (const int32_t*)r.operand(v[6], na, 4);
    const int32_t* b = (const int32_t*)r.operand(v[7], nnz, 4);
    void* const vals = r.operand(v[8], nnz, e);
    void* const in = r.operand(v[9], nnz > 0 ? r.times(n, kk) : 0, e);
    void* const out = r.operand(v[10], r.times(atleast0(m), kk), e);
    void* const stream = r.stream(v[14]);
    if (!r.ok) return -1;
    return unlocked([&]() -> int {
      return k == 0 ? ((decltype(&spmv_csr))fn)(m, n, nnz, a, b, vals, in, out, alpha, beta, dtype, stream)
                    : ((decltype(&spmm_csr))fn)(m, n, nnz, k, a, b, vals, in, out, alpha, beta, dtype, stream);
    });
  });
}

// (fn, m, n, width, k, col_ids, vals, in, out, alpha, beta, dtype, stream); k == 0: SpMV.
PyObject* ell_product(PyObject*, PyObject* const* v, Py_ssize_t argc) {
  return guarded([&]() -> int {
    if (argc != 13) return -1;
    Reader r;
    void* const fn = r.address(v[0]);
    const int64_t m = r.size(v[1]), n = r.size(v[2]), width = r.size(v[3]), k = r.size(v[4]);
    const float alpha = r.scalar(v[9]), beta = r.scalar(v[10]);
    const int dtype = r.dtype(v[11]);
    if (!r.ok || k < 0) return -1;
    const int64_t e = dtype == B200SP_F32 ? 4 : 2, kk = k > 1 ? k : 1, slots = r.times(m, width);
    const int32_t* cols = (const int32_t*)r.operand(v[5], slots, 4);
    void* const vals = r.operand(v[6], slots, e);
    void* const in = r.operand(v[7], slots > 0 ? r.times(n, kk) : 0, e);
    void* const out = r.operand(v[8], r.times(m, kk), e);
    void* const stream = r.stream(v[12]);
    if (!r.ok) return -1;
    return unlocked([&]() -> int {
      return k == 0 ? ((decltype(&spmv_ell))fn)(m, n, width, cols, vals, in, out, alpha, beta, dtype, stream)
                    : ((decltype(&spmm_ell))fn)(m, n, width, k, cols, vals, in, out, alpha, beta, dtype, stream);
    });
  });
}

// (info fn, fn, plan, k, col_idx, vals, in, out, alpha, beta, dtype, stream); k == 0: SpMV.
PyObject* plan_product(PyObject*, PyObject* const* v, Py_ssize_t argc) {
  return guarded([&]() -> int {
    if (argc != 12) return -1;
    Reader r;
    void* const info = r.address(v[0]);
    void* const fn = r.address(v[1]);
    b200sp_plan* const plan = (b200sp_plan*)r.address(v[2]);
    const int64_t k = r.size(v[3]);
    const float alpha = r.scalar(v[8]), beta = r.scalar(v[9]);
    const int dtype = r.dtype(v[10]);
    if (!r.ok || k < 0) return -1;
    b200sp_plan_info_t I;
    const int rc = ((decltype(&b200sp_plan_info))info)(plan, &I);
    if (rc != B200SP_OK) return -1;
    const int64_t e = dtype == B200SP_F32 ? 4 : 2, kk = k > 1 ? k : 1;
    const int32_t* col = (const int32_t*)r.operand(v[4], I.nnz, 4);
    void* const vals = r.operand(v[5], I.nnz, e);
    void* const in = r.operand(v[6], I.nnz > 0 ? r.times(I.n, kk) : 0, e);
    void* const out = r.operand(v[7], r.times(I.m, kk), e);
    void* const stream = r.stream(v[11]);
    if (!r.ok) return -1;
    return unlocked([&]() -> int {
      return k == 0 ? ((decltype(&b200sp_spmv))fn)(plan, col, vals, in, out, alpha, beta, dtype, stream)
                    : ((decltype(&b200sp_spmm))fn)(plan, k, col, vals, in, out, alpha, beta, dtype, stream);
    });
  });
}

// (fn, m, n, nnz, row_ptr, stream): the new plan's address, or -1 / -2 - status (a plan's address is never negative as a signed number).
PyObject* plan_create(PyObject*, PyObject* const* v, Py_ssize_t argc) {
  long long result = -1;
  try {
    if (argc == 6) {
      Reader r;
      void* const fn = r.address(v[0]);
      const int64_t m = r.size(v[1]), n = r.size(v[2]), nnz = r.size(v[3]);
      const int32_t* row_ptr = (const int32_t*)r.operand(v[4], m > 0 ? r.plus1(m) : 0, 4);
      void* const stream = r.stream(v[5]);
      if (r.ok) {
        b200sp_plan* plan = nullptr;
        const int status = unlocked([&]() -> int { return ((decltype(&b200sp_plan_create))fn)(&plan, m, n, nnz, row_ptr, stream); });
        result = status == B200SP_OK ? (long long)(intptr_t)plan : -2 - status;
      }
    }
  } catch (...) {
    result = -1;
  }
  return PyLong_FromLongLong(result);
}

PyMethodDef methods[] = {
    {"plan_create", (PyCFunction)(void (*)(void))plan_create, METH_FASTCALL, nullptr},
    {"product", (PyCFunction)(void (*)(void))product, METH_FASTCALL, nullptr},
    {"ell_product", (PyCFunction)(void (*)(void))ell_product, METH_FASTCALL, nullptr},
    {"plan_product", (PyCFunction)(void (*)(void))plan_product, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_marshal", "Native argument marshalling of the b200sp binding.", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" PyObject* PyInit__marshal() { return PyModule_Create(&module_def); }
