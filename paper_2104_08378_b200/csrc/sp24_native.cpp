// Native form of the binding's short calls (a Python extension module over torch's C++ API): argument marshalling, the
// allocation of the result, and the call of the C ABI.  For a small product the marshalling in Python costs more than the
// kernel takes (f16 256 x 256 x 512: 9.9 us of host time a call for 3.2 us on the device; 2.9 of it the allocation through
// torch's Python layer, 3 the marshalling, 1 ctypes, 3.1 the launch); here the call takes 4.5 us, 2.8 with the result given.
//
// Every function takes what the Python one has been given and returns None if anything about it is out of the ordinary
// (another type than a plain CUDA tensor, an active torch-function mode, a type or shape that the Python form rejects, no
// workspace yet, an exception from torch): the Python form then deals with the call from the start.  Otherwise it
// returns the result, or the status as an int if the library refused the call.  The interpreter lock is released around
// the allocation and the call, as torch and ctypes do.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <ATen/ops/empty.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "sp24.h"

namespace {

const at::ScalarType kScalar[7] = {at::kHalf, at::kBFloat16, at::kChar, at::kFloat, at::kInt, at::kFloat8_e4m3fn, at::kFloat8_e5m2};
const char* const kName[7] = {"f16", "bf16", "i8", "f32", "i32", "e4m3", "e5m2"};

// sp24_dtype of a torch type, of a type's name (-1: none)
int type_code(at::ScalarType t) {
  for (int i = 0; i < 7; ++i)
    if (kScalar[i] == t) return i;
  return -1;
}
int type_code(PyObject* name) {
  if (!PyUnicode_CheckExact(name)) return -1;
  for (int i = 0; i < 7; ++i)
    if (PyUnicode_CompareWithASCIIString(name, kName[i]) == 0) return i;
  return -1;
}

// A torch.Tensor itself (no subclass, no wrapper of a transform) in CUDA memory with at least `dims` dimensions, else null.
const at::Tensor* plain(PyObject* o, int64_t dims) {
  if (!THPVariable_CheckExact(o)) return nullptr;
  const at::Tensor& t = THPVariable_Unpack(o);
  const c10::DispatchKeySet keys = t.key_set();
  if (!t.is_cuda() || t.layout() != at::kStrided || t.dim() < dims || !t.has_storage() || t.is_conj() || t.is_neg() ||
      keys.has(c10::DispatchKey::Functionalize) || keys.has(c10::DispatchKey::Python))
    return nullptr;
  return &t;
}

// data_ptr() of an optional tensor; false: not an ordinary one
bool pointer(PyObject* o, const void** p) {
  if (o == Py_None) {
    *p = nullptr;
    return true;
  }
  const at::Tensor* t = plain(o, 0);
  if (t == nullptr) return false;
  *p = t->data_ptr();
  return true;
}

// an ordinary Python number
bool number(PyObject* o, double* v) {
  if (PyFloat_CheckExact(o)) {
    *v = PyFloat_AS_DOUBLE(o);
    return true;
  }
  return false;
}

struct Stream {
  cudaStream_t handle;
  Stream() : handle(c10::cuda::getCurrentCUDAStream().stream()) {}
};

// The workspace: the caller's, or the one kept for the device and stream.
bool workspace(PyObject* kept, PyObject* ws, const at::Tensor& a, cudaStream_t stream, void** p, size_t* bytes) {
  if (ws == Py_None) {
    PyObject* key = Py_BuildValue("(iN)", (int)a.get_device(), PyLong_FromUnsignedLongLong((unsigned long long)(uintptr_t)stream));
    if (key == nullptr) return false;
    ws = PyDict_GetItemWithError(kept, key);
    Py_DECREF(key);
    if (ws == nullptr) return false;
  }
  const at::Tensor* t = plain(ws, 0);
  if (t == nullptr) return false;
  *p = t->data_ptr();
  *bytes = (size_t)t->numel();
  return true;
}

PyObject* none() {
  PyErr_Clear();
  Py_RETURN_NONE;
}

// What the three products share: A, the result's type and place, C, the orders.
struct Product {
  const at::Tensor* a = nullptr;
  sp24_gemm_desc d = {};
  const void *meta = nullptr, *c = nullptr;
  void* ws = nullptr;
  size_t ws_bytes = 0;
  cudaStream_t stream = nullptr;
  bool cols = false;

  bool init(PyObject* A, PyObject* meta_, int ab, PyObject* cd, PyObject* dense, PyObject* b_rows, PyObject* cd_cols) {
    if (at::impl::torch_function_mode_enabled()) return false;
    a = plain(A, 2);
    if (a == nullptr || !pointer(meta_, &meta)) return false;
    if (ab < 0) ab = type_code(a->scalar_type());
    int out = cd == Py_None ? (ab == SP24_I8 ? SP24_I32 : (ab == SP24_E4M3 || ab == SP24_E5M2 ? SP24_BF16 : ab)) : type_code(cd);
    if (ab < 0 || out < 0) return false;
    cols = cd_cols == Py_True;
    if ((dense != Py_True && dense != Py_False) || (b_rows != Py_True && b_rows != Py_False) || (!cols && cd_cols != Py_False)) return false;
    d.ab_type = (sp24_dtype)ab;
    d.cd_type = (sp24_dtype)out;
    d.a_is_dense = dense == Py_True;
    d.M = a->size(0);
    d.K = d.a_is_dense ? a->size(1) : 2 * a->size(1);
    d.lda = a->stride(0);
    d.order_b = b_rows == Py_True ? SP24_ROW_MAJOR : SP24_COL_MAJOR;
    d.order_c = d.order_d = cols ? SP24_COL_MAJOR : SP24_ROW_MAJOR;
    return true;
  }
  // N and K are set: C, the workspace, and the call with the result's pointer
  template <typename Call>
  PyObject* run(PyObject* kept, PyObject* C, PyObject* out, PyObject* ws_, Call call) {
    d.ldc = cols ? d.M : d.N;
    if (C != Py_None) {
      const at::Tensor* t = plain(C, 1);
      if (t == nullptr) return none();
      d.ldc = t->stride(0);
      c = t->data_ptr();
    }
    stream = Stream().handle;
    if (!workspace(kept, ws_, *a, stream, &ws, &ws_bytes)) return none();
    const void* A = a->data_ptr();
    at::Tensor made;
    void* D = nullptr;
    if (out == Py_None) {
      d.ldd = cols ? d.M : d.N;
    } else {
      const at::Tensor* t = plain(out, 1);
      if (t == nullptr) return none();
      d.ldd = t->stride(0);
      D = t->data_ptr();
    }
    int status;
    {
      pybind11::gil_scoped_release unlocked;
      if (out == Py_None) {
        made = at::empty({cols ? d.N : d.M, cols ? d.M : d.N}, a->options().dtype(kScalar[d.cd_type]));
        if (d.ldd < 1) d.ldd = 1;  // (as torch reports the stride of an empty tensor)
        D = made.data_ptr();
      }
      status = call(*this, A, D);
    }
    if (status != SP24_OK) return PyLong_FromLong(status);
    if (out == Py_None) return THPVariable_Wrap(std::move(made));
    Py_INCREF(out);
    return out;
  }
};

template <typename F>
F function(PyObject* address) {
  return reinterpret_cast<F>(PyLong_AsVoidPtr(address));
}

// gemm(address, workspaces, A, meta, Bt, alpha, beta, C, out, cd, a_is_dense, ws, b_row_major, cd_col_major)
PyObject* gemm(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (n != 14) return none();
  try {
    Product p;
    double alpha, beta;
    if (!p.init(v[2], v[3], -1, v[9], v[10], v[12], v[13])) return none();
    const at::Tensor* b = plain(v[4], 2);
    if (b == nullptr || !number(v[5], &alpha)) return none();
    if (PyLong_CheckExact(v[6]) && p.d.ab_type == SP24_I8) beta = (double)PyLong_AsLong(v[6]);
    else if (!number(v[6], &beta)) return none();
    const bool rows = p.d.order_b == SP24_ROW_MAJOR, whole = p.d.ab_type == SP24_I8;
    if (b->size(rows ? 0 : 1) != p.d.K) return none();
    if (whole && (alpha != 1.0 || (beta != 0.0 && beta != 1.0))) return none();
    p.d.N = b->size(rows ? 1 : 0);
    p.d.ldb = b->stride(0);
    const void* B = b->data_ptr();
    const auto fn = function<decltype(&sp24_gemm)>(v[0]);
    return p.run(v[1], v[7], v[8], v[11], [&](const Product& q, const void* A, void* D) {
      const float fa = (float)alpha, fb = (float)beta;
      const int32_t ia = 1, ib = (int32_t)(whole ? beta : 0.0);
      return (int)fn(&q.d, whole ? (const void*)&ia : &fa, A, q.meta, B, whole ? (const void*)&ib : &fb, q.c, D, q.ws, q.ws_bytes, q.stream);
    });
  } catch (...) {
    return none();
  }
}

// gemm_i8_dequant(address, workspaces, A, meta, Bt, row_scale, bias, relu, out_scale, cd, out, a_is_dense, ws, b_row_major,
// cd_col_major)
PyObject* gemm_i8_dequant(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (n != 15) return none();
  try {
    Product p;
    double out_scale;
    if (v[9] == Py_None || !p.init(v[2], v[3], SP24_I8, v[9], v[11], v[13], v[14])) return none();
    const at::Tensor* b = plain(v[4], 2);
    const void *scale, *bias;
    if (b == nullptr || !pointer(v[5], &scale) || !pointer(v[6], &bias) || !number(v[8], &out_scale)) return none();
    const int relu = PyObject_IsTrue(v[7]);
    if (relu < 0) return none();
    p.d.N = b->size(p.d.order_b == SP24_ROW_MAJOR ? 1 : 0);
    p.d.ldb = b->stride(0);
    const void* B = b->data_ptr();
    const auto fn = function<decltype(&sp24_gemm_i8_dequant)>(v[0]);
    return p.run(v[1], Py_None, v[10], v[12], [&](const Product& q, const void* A, void* D) {
      return (int)fn(&q.d, A, q.meta, B, (const float*)scale, (const float*)bias, relu, (float)out_scale, D, q.ws, q.ws_bytes, q.stream);
    });
  } catch (...) {
    return none();
  }
}

// conv3x3_nhwc(address, workspaces, A, meta, x, alpha, beta, C, out, cd, a_is_dense, ws, nhwc_out)
PyObject* conv3x3_nhwc(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (n != 13) return none();
  try {
    Product p;
    double alpha, beta;
    if (!p.init(v[2], v[3], -1, v[9], v[10], Py_False, v[12])) return none();
    const at::Tensor* x = plain(v[4], 4);
    if (x == nullptr || x->dim() != 4 || p.d.ab_type == SP24_I8 || !number(v[5], &alpha) || !number(v[6], &beta)) return none();
    const int64_t nb = x->size(0), h = x->size(1), w = x->size(2), cin = x->size(3);
    p.d.K = p.d.ldb = 9 * cin;
    p.d.N = nb * h * w;
    const void* X = x->data_ptr();
    const auto fn = function<decltype(&sp24_conv3x3_nhwc)>(v[0]);
    return p.run(v[1], v[7], v[8], v[11], [&](const Product& q, const void* A, void* D) {
      const float fa = (float)alpha, fb = (float)beta;
      return (int)fn(&q.d, nb, h, w, cin, &fa, A, q.meta, X, &fb, q.c, D, q.ws, q.ws_bytes, q.stream);
    });
  } catch (...) {
    return none();
  }
}

// compress(address, address of sp24_meta_bytes, x, layout) -> (vals, meta, None)
PyObject* compress(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (n != 4 || !PyLong_CheckExact(v[3]) || at::impl::torch_function_mode_enabled()) return none();
  try {
    const at::Tensor* x = plain(v[2], 2);
    if (x == nullptr || x->dim() != 2) return none();
    const int dt = type_code(x->scalar_type());
    const long layout = PyLong_AsLong(v[3]);
    if (dt < 0 || (layout != 0 && layout != 1)) return none();
    const int64_t M = x->size(0), K = x->size(1);
    const auto fn = function<decltype(&sp24_compress)>(v[0]);
    const auto bytes = function<decltype(&sp24_meta_bytes)>(v[1]);
    const cudaStream_t stream = Stream().handle;
    const void* X = x->data_ptr();
    at::Tensor vals, meta;
    int status;
    {
      pybind11::gil_scoped_release unlocked;
      vals = at::empty({M, K / 2}, x->options());
      meta = at::empty({(int64_t)bytes((sp24_dtype)dt, M, K, (sp24_meta_layout)layout)}, x->options().dtype(at::kByte));
      status = (int)fn((sp24_dtype)dt, M, K, X, M > 1 ? x->stride(0) : K, vals.data_ptr(), K / 2, meta.data_ptr(),
                       (sp24_meta_layout)layout, nullptr, stream);
    }
    if (status != SP24_OK) return PyLong_FromLong(status);
    return Py_BuildValue("(NNO)", THPVariable_Wrap(std::move(vals)), THPVariable_Wrap(std::move(meta)), Py_None);
  } catch (...) {
    return none();
  }
}

// apply_mask(address, w, meta, layout, out) -> out
PyObject* apply_mask(PyObject*, PyObject* const* v, Py_ssize_t n) {
  if (n != 5 || !PyLong_CheckExact(v[3]) || at::impl::torch_function_mode_enabled()) return none();
  try {
    const at::Tensor *w = plain(v[1], 2), *out = plain(v[4], 1);
    const void* meta;
    if (w == nullptr || w->dim() != 2 || out == nullptr || !pointer(v[2], &meta)) return none();
    const int dt = type_code(w->scalar_type());
    const long layout = PyLong_AsLong(v[3]);
    if (dt < 0 || (layout != 0 && layout != 1)) return none();
    const int64_t M = w->size(0), K = w->size(1);
    const auto fn = function<decltype(&sp24_apply_mask)>(v[0]);
    const cudaStream_t stream = Stream().handle;
    const void* W = w->data_ptr();
    void* Y = out->data_ptr();
    const int64_t ldw = M > 1 ? w->stride(0) : K, ldy = M > 1 ? out->stride(0) : K;
    int status;
    {
      pybind11::gil_scoped_release unlocked;
      status = (int)fn((sp24_dtype)dt, M, K, W, ldw, meta, (sp24_meta_layout)layout, Y, ldy, stream);
    }
    if (status != SP24_OK) return PyLong_FromLong(status);
    Py_INCREF(v[4]);
    return v[4];
  } catch (...) {
    return none();
  }
}

#define SP24_METHOD(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {SP24_METHOD(gemm), SP24_METHOD(gemm_i8_dequant), SP24_METHOD(conv3x3_nhwc), SP24_METHOD(compress),
                         SP24_METHOD(apply_mask), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native() { return PyModule_Create(&module); }
