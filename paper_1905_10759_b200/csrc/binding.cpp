// The entry points that a program calls once per layer and pass, as native functions: a call of a few microseconds spent more
// than a third of its host time marshalling its arguments in Python (hbmm_quantize of a 1 x 4096 row: 5.0 us, of which the
// library, its checks and the launch included, takes 3.2).  Names, arguments, defaults, checks and errors are those of the
// Python functions they stand for; the C functions of libhbmm.so are handed over as addresses when hbmm.py is imported, and
// run without the interpreter lock, as ctypes runs them.
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/Exceptions.h>
#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include "hbmm.h"

namespace {

decltype(&hbmm_quantize) f_quantize;
decltype(&hbmm_gemm) f_gemm;
decltype(&hbmm_gemm_ex) f_gemm_ex;
decltype(&hbmm_conv_im2col_ex) f_conv;
decltype(&hbmm_conv_im2col_fused) f_conv_fused;
decltype(&hbmm_binarize_dense) f_dense;
decltype(&hbmm_binarize_backward) f_backward;
PyObject* g_error;                 // HbmmError
PyTypeObject *t_operand, *t_geom, *t_epilogue;      // the ctypes structures that stand for hbmm_operand, hbmm_conv_geom, hbmm_epilogue
PyObject *s_desc, *s_cuda_stream;

// Arguments of a METH_FASTCALL | METH_KEYWORDS call in the order of `names`; absent ones stay null.
bool take(const char* what, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames, const char* const* names, int n, int required, PyObject** out) {
  if (nargs > n) {
    PyErr_Format(PyExc_TypeError, "%s() takes at most %d positional arguments (%zd given)", what, n, nargs);
    return false;
  }
  for (int i = 0; i < n; i++) out[i] = i < nargs ? args[i] : nullptr;
  const Py_ssize_t nk = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
  for (Py_ssize_t k = 0; k < nk; k++) {
    PyObject* key = PyTuple_GET_ITEM(kwnames, k);
    int at = 0;
    while (at < n && PyUnicode_CompareWithASCIIString(key, names[at]) != 0) at++;
    if (at == n) {
      PyErr_Format(PyExc_TypeError, "%s() got an unexpected keyword argument '%U'", what, key);
      return false;
    }
    if (out[at]) {
      PyErr_Format(PyExc_TypeError, "%s() got multiple values for argument '%s'", what, names[at]);
      return false;
    }
    out[at] = args[nargs + k];
  }
  for (int i = 0; i < required; i++)
    if (!out[i]) {
      PyErr_Format(PyExc_TypeError, "%s() missing required argument '%s'", what, names[i]);
      return false;
    }
  return true;
}

const at::Tensor* tensor_of(PyObject* o) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "a torch.Tensor is expected, got %s", Py_TYPE(o)->tp_name);
    return nullptr;
  }
  return &THPVariable_Unpack(o);
}
bool none(PyObject* o) { return !o || o == Py_None; }

bool device_ptr(const at::Tensor& t, void** p) {
  if (!t.is_cuda()) {
    PyErr_SetString(PyExc_ValueError, "device tensor expected");
    return false;
  }
  *p = t.data_ptr();
  return true;
}
bool dtype_code(const at::Tensor& t, int32_t* code) {
  const at::ScalarType s = t.scalar_type();
  if (s == at::kFloat) { *code = HBMM_F32; return true; }
  if (s == at::kBFloat16) { *code = HBMM_BF16; return true; }
  PyErr_Format(PyExc_TypeError, "only float32 and bfloat16 tensors are accepted, got torch.%s", c10::toString(s));
  return false;
}
bool integer(PyObject* o, long long* v) {
  *v = PyLong_AsLongLong(o);
  return !(*v == -1 && PyErr_Occurred());
}
bool small_integer(PyObject* o, int32_t* v) {
  long long w;
  if (!integer(o, &w)) return false;
  *v = static_cast<int32_t>(w);               // as ctypes passes it on
  return true;
}
// The bytes behind a ctypes structure, of the type it is declared as and no other: what they hold is taken for sizes and addresses.
template <typename T>
struct Struct {
  Py_buffer view{};
  const T* p = nullptr;
  ~Struct() { if (view.obj) PyBuffer_Release(&view); }
  bool open(PyObject* o, PyTypeObject* type) {
    if (!PyObject_TypeCheck(o, type)) {
      PyErr_Format(PyExc_TypeError, "%s expected, got %s", type->tp_name, Py_TYPE(o)->tp_name);
      return false;
    }
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) return false;
    if (view.len < static_cast<Py_ssize_t>(sizeof(T))) {
      PyErr_Format(PyExc_TypeError, "%s is shorter than the library's", type->tp_name);
      return false;
    }
    p = static_cast<const T*>(view.buf);
    return true;
  }
  bool open_desc(PyObject* operand) {
    PyObject* d = PyObject_GetAttr(operand, s_desc);
    if (!d) return false;
    const bool ok = open(d, t_operand);
    Py_DECREF(d);                             // the view holds it
    return ok;
  }
};
bool stream_of(PyObject* o, void** s) {
  if (none(o)) {
    *s = c10::cuda::getCurrentCUDAStream().stream();
    return true;
  }
  PyObject* h = PyObject_GetAttr(o, s_cuda_stream);
  if (!h) return false;
  const unsigned long long v = PyLong_AsUnsignedLongLong(h);
  Py_DECREF(h);
  if (v == static_cast<unsigned long long>(-1) && PyErr_Occurred()) return false;
  *s = reinterpret_cast<void*>(static_cast<uintptr_t>(v));
  return true;
}
struct Owned {                     // one reference, given back at the end
  PyObject* o;
  ~Owned() { Py_XDECREF(o); }
};
struct Buffer {
  void* p = nullptr;
  size_t bytes = 0;
  bool open(PyObject* o) {                    // None: no workspace
    if (none(o)) return true;
    const at::Tensor* t = tensor_of(o);
    if (!t || !device_ptr(*t, &p)) return false;
    bytes = t->nbytes();
    return true;
  }
};
PyObject* done(int32_t status, const char* where, PyObject* result) {
  if (status != HBMM_OK) {
    PyObject* e = PyObject_CallFunction(g_error, "is", static_cast<int>(status), where);
    if (e) {
      PyErr_SetObject(g_error, e);
      Py_DECREF(e);
    }
    return nullptr;
  }
  Py_INCREF(result);
  return result;
}
#define HBMM_CALL(expr)            \
  int32_t status;                  \
  Py_BEGIN_ALLOW_THREADS;          \
  status = (expr);                 \
  Py_END_ALLOW_THREADS

PyObject* py_quantize(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kw) {
  HANDLE_TH_ERRORS
  static const char* const names[] = {"x", "out", "stream"};
  PyObject* a[3];
  if (!take("quantize", args, nargs, kw, names, 3, 2, a)) return nullptr;
  const at::Tensor* x = tensor_of(a[0]);
  if (!x) return nullptr;
  if (x->dim() != 2 || x->stride(1) != 1) {
    PyErr_SetString(PyExc_ValueError, "x must be a row-major 2-D tensor");
    return nullptr;
  }
  void *p, *s;
  int32_t dt;
  Struct<hbmm_operand> out;
  if (!out.open_desc(a[1]) || !device_ptr(*x, &p) || !dtype_code(*x, &dt) || !stream_of(a[2], &s)) return nullptr;
  const int64_t rows = x->size(0), K = x->size(1), ld = x->stride(0);
  HBMM_CALL(f_quantize(p, dt, rows, K, ld, out.p, s));
  return done(status, "hbmm_quantize", a[1]);
  END_HANDLE_TH_ERRORS
}

PyObject* gemm_any(const char* what, const char* where, bool ex, PyObject** a, PyObject* path_o, PyObject* ws_o, PyObject* stream_o) {
  Buffer ws;
  Struct<hbmm_operand> A, W;
  void *c, *s;
  int32_t path = HBMM_PATH_AUTO;
  if (!ws.open(ws_o) || !A.open_desc(a[0]) || !W.open_desc(a[1])) return nullptr;
  const at::Tensor* C = tensor_of(a[2]);
  if (!C || !device_ptr(*C, &c) || (ex && !small_integer(path_o, &path)) || !stream_of(stream_o, &s)) return nullptr;
  const int64_t ldc = C->stride(0);
  HBMM_CALL(ex ? f_gemm_ex(A.p, W.p, static_cast<float*>(c), ldc, ws.p, ws.bytes, path, s) : f_gemm(A.p, W.p, static_cast<float*>(c), ldc, ws.p, ws.bytes, s));
  return done(status, where, a[2]);
}
PyObject* py_gemm(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kw) {
  HANDLE_TH_ERRORS
  static const char* const names[] = {"A", "W", "C", "workspace", "stream"};
  PyObject* a[5];
  if (!take("gemm", args, nargs, kw, names, 5, 3, a)) return nullptr;
  return gemm_any("gemm", "hbmm_gemm", false, a, nullptr, a[3], a[4]);
  END_HANDLE_TH_ERRORS
}
PyObject* py_gemm_ex(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kw) {
  HANDLE_TH_ERRORS
  static const char* const names[] = {"A", "W", "C", "path", "workspace", "stream"};
  PyObject* a[6];
  if (!take("gemm_ex", args, nargs, kw, names, 6, 4, a)) return nullptr;
  return gemm_any("gemm_ex", "hbmm_gemm_ex", true, a, a[3], a[4], a[5]);
  END_HANDLE_TH_ERRORS
}

PyObject* py_conv_im2col(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kw) {
  HANDLE_TH_ERRORS
  static const char* const names[] = {"x", "geom", "beta_a", "a_scale_dtype", "W", "C_out", "workspace", "stream", "flags"};
  PyObject* a[9];
  if (!take("conv_im2col", args, nargs, kw, names, 9, 7, a)) return nullptr;
  const at::Tensor* x = tensor_of(a[0]);
  if (!x) return nullptr;
  if (!x->is_contiguous()) {
    PyErr_SetString(PyExc_ValueError, "x must be a contiguous NCHW tensor");
    return nullptr;
  }
  void *p, *c = nullptr, *s;
  int32_t dt, beta, sdt;
  long long flags = 0;
  int64_t ldc = 0;
  Struct<hbmm_conv_geom> geom;
  Struct<hbmm_operand> W;
  Buffer ws;
  if (!geom.open(a[1], t_geom) || !W.open_desc(a[4]) || !device_ptr(*x, &p) || !dtype_code(*x, &dt) || !small_integer(a[2], &beta) ||
      !small_integer(a[3], &sdt) || (!none(a[8]) && !integer(a[8], &flags)))
    return nullptr;
  if (!none(a[5])) {
    const at::Tensor* C = tensor_of(a[5]);
    if (!C || !device_ptr(*C, &c)) return nullptr;
    ldc = C->stride(0);
  }
  if (!ws.open(a[6]) || !stream_of(a[7], &s)) return nullptr;
  HBMM_CALL(f_conv(p, dt, geom.p, beta, sdt, W.p, static_cast<float*>(c), ldc, ws.p, ws.bytes, static_cast<uint32_t>(flags), s));
  return done(status, flags ? "hbmm_conv_im2col_ex" : "hbmm_conv_im2col", a[5]);
  END_HANDLE_TH_ERRORS
}

PyObject* py_conv_im2col_fused(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kw) {
  HANDLE_TH_ERRORS
  static const char* const names[] = {"x", "geom", "beta_a", "a_scale_dtype", "W", "ep", "workspace", "stream", "flags"};
  PyObject* a[9];
  if (!take("conv_im2col_fused", args, nargs, kw, names, 9, 7, a)) return nullptr;
  const at::Tensor* x = tensor_of(a[0]);
  if (!x) return nullptr;
  if (!x->is_contiguous()) {
    PyErr_SetString(PyExc_ValueError, "x must be contiguous");
    return nullptr;
  }
  void *p, *s;
  int32_t dt, beta, sdt;
  long long flags = 0;
  Struct<hbmm_conv_geom> geom;
  Struct<hbmm_operand> W;
  Struct<hbmm_epilogue> ep;
  Buffer ws;
  if (!geom.open(a[1], t_geom) || !W.open_desc(a[4]) || !ep.open(a[5], t_epilogue) || !device_ptr(*x, &p) || !dtype_code(*x, &dt) ||
      !small_integer(a[2], &beta) || !small_integer(a[3], &sdt) || !ws.open(a[6]) || !stream_of(a[7], &s) || (a[8] && !integer(a[8], &flags)))
    return nullptr;
  HBMM_CALL(f_conv_fused(p, dt, geom.p, beta, sdt, W.p, ep.p, ws.p, ws.bytes, static_cast<uint32_t>(flags), s));
  return done(status, "hbmm_conv_im2col_fused", Py_None);
  END_HANDLE_TH_ERRORS
}

PyObject* py_binarize_backward(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kw) {
  HANDLE_TH_ERRORS
  static const char* const names[] = {"x", "gy", "beta", "gx", "stream"};
  PyObject* a[5];
  if (!take("binarize_backward", args, nargs, kw, names, 5, 3, a)) return nullptr;
  const at::Tensor *x = tensor_of(a[0]), *gy = x ? tensor_of(a[1]) : nullptr;
  if (!gy) return nullptr;
  if (x->scalar_type() != at::kFloat || gy->scalar_type() != at::kFloat || x->sizes() != gy->sizes() || x->dim() != 2) {
    PyErr_SetString(PyExc_ValueError, "x and gy must be fp32 matrices of one shape");
    return nullptr;
  }
  if (x->stride(1) != 1 || gy->stride(1) != 1) {
    PyErr_SetString(PyExc_ValueError, "rows must be contiguous");
    return nullptr;
  }
  at::Tensor own;
  PyObject* result = a[3];
  if (none(result)) {
    own = at::empty(x->sizes(), at::TensorOptions().dtype(at::kFloat).device(x->device()));
    result = THPVariable_Wrap(own);
    if (!result) return nullptr;
  } else {
    Py_INCREF(result);
  }
  const Owned keep{result};
  const at::Tensor* gx = tensor_of(result);
  void *px, *pg, *po, *s;
  int32_t beta;
  if (!gx || !device_ptr(*x, &px) || !device_ptr(*gy, &pg) || !small_integer(a[2], &beta) || !device_ptr(*gx, &po) || !stream_of(a[4], &s)) return nullptr;
  const int64_t ldx = x->stride(0), ldg = gy->stride(0), rows = x->size(0), K = x->size(1), ldo = gx->stride(0);
  HBMM_CALL(f_backward(static_cast<const float*>(px), ldx, static_cast<const float*>(pg), ldg, rows, K, beta, static_cast<float*>(po), ldo, s));
  return done(status, "hbmm_binarize_backward", result);
  END_HANDLE_TH_ERRORS
}

PyObject* py_binarize_dense(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kw) {
  HANDLE_TH_ERRORS
  static const char* const names[] = {"x", "beta", "out_dtype", "out", "stream"};
  PyObject* a[5];
  if (!take("binarize_dense", args, nargs, kw, names, 5, 2, a)) return nullptr;
  const at::Tensor* x = tensor_of(a[0]);
  if (!x) return nullptr;
  if (x->scalar_type() != at::kFloat || x->dim() != 2 || x->stride(1) != 1) {
    PyErr_SetString(PyExc_ValueError, "x must be an fp32 matrix with contiguous rows");
    return nullptr;
  }
  int32_t beta, out_code = HBMM_F32;
  if ((a[2] && !small_integer(a[2], &out_code)) || !small_integer(a[1], &beta)) return nullptr;
  const at::ScalarType tdt = out_code == HBMM_BF16 ? at::kBFloat16 : at::kFloat;
  PyObject* result = a[3];
  if (none(result)) {
    at::Tensor own = at::empty(x->sizes(), at::TensorOptions().dtype(tdt).device(x->device()));
    result = THPVariable_Wrap(own);
    if (!result) return nullptr;
  } else {
    Py_INCREF(result);
  }
  const Owned keep{result};
  const at::Tensor* out = tensor_of(result);
  if (!out) return nullptr;
  if (out->scalar_type() != tdt || out->sizes() != x->sizes() || out->stride(1) != 1) {
    PyErr_SetString(PyExc_ValueError, "out must match x's shape and the requested type");
    return nullptr;
  }
  void *px, *po, *s;
  if (!device_ptr(*x, &px) || !device_ptr(*out, &po) || !stream_of(a[4], &s)) return nullptr;
  const int64_t ldx = x->stride(0), rows = x->size(0), K = x->size(1), ldo = out->stride(0);
  HBMM_CALL(f_dense(static_cast<const float*>(px), ldx, rows, K, beta, po, out_code, ldo, s));
  return done(status, "hbmm_binarize_dense", result);
  END_HANDLE_TH_ERRORS
}

// connect(HbmmError, hbmm_operand, hbmm_conv_geom, hbmm_epilogue, addresses of the C functions in the order of the f_ pointers above)
PyObject* py_connect(PyObject*, PyObject* args) {
  PyObject *err, *types[3];
  unsigned long long p[7];
  if (!PyArg_ParseTuple(args, "OO!O!O!KKKKKKK", &err, &PyType_Type, &types[0], &PyType_Type, &types[1], &PyType_Type, &types[2], &p[0], &p[1],
                        &p[2], &p[3], &p[4], &p[5], &p[6]))
    return nullptr;
  f_quantize = reinterpret_cast<decltype(f_quantize)>(p[0]);
  f_gemm = reinterpret_cast<decltype(f_gemm)>(p[1]);
  f_gemm_ex = reinterpret_cast<decltype(f_gemm_ex)>(p[2]);
  f_conv = reinterpret_cast<decltype(f_conv)>(p[3]);
  f_conv_fused = reinterpret_cast<decltype(f_conv_fused)>(p[4]);
  f_dense = reinterpret_cast<decltype(f_dense)>(p[5]);
  f_backward = reinterpret_cast<decltype(f_backward)>(p[6]);
  Py_INCREF(err);
  Py_XSETREF(g_error, err);
  PyTypeObject** const held[] = {&t_operand, &t_geom, &t_epilogue};
  for (int i = 0; i < 3; i++) {
    Py_INCREF(types[i]);
    Py_XSETREF(*held[i], reinterpret_cast<PyTypeObject*>(types[i]));
  }
  Py_RETURN_NONE;
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL | METH_KEYWORDS
PyMethodDef methods[] = {
    {"quantize", FAST(py_quantize),
     "quantize($module, /, x, out, stream=None)\n--\n\nhbmm_quantize: Hadamard-binarize and pack the rows of ``x`` [rows, K] into ``out``."},
    {"gemm", FAST(py_gemm),
     "gemm($module, /, A, W, C, workspace=None, stream=None)\n--\n\nhbmm_gemm: C[M, N] (fp32, row-major, caller-allocated) = A~ W~^T."},
    {"gemm_ex", FAST(py_gemm_ex),
     "gemm_ex($module, /, A, W, C, path, workspace=None, stream=None)\n--\n\nhbmm_gemm_ex: hbmm_gemm on the path asked for."},
    {"conv_im2col", FAST(py_conv_im2col),
     "conv_im2col($module, /, x, geom, beta_a, a_scale_dtype, W, C_out, workspace, stream=None, flags=0)\n--\n\n"
     "hbmm_conv_im2col (flags == 0) / hbmm_conv_im2col_ex: x NCHW contiguous; C_out fp32 [B*Ho*Wo, N]."},
    {"conv_im2col_fused", FAST(py_conv_im2col_fused),
     "conv_im2col_fused($module, /, x, geom, beta_a, a_scale_dtype, W, ep, workspace, stream=None, flags=0)\n--\n\n"
     "hbmm_conv_im2col_fused: x NCHW contiguous (or NHWC bf16 with CONV_INPUT_NHWC)."},
    {"binarize_dense", FAST(py_binarize_dense),
     "binarize_dense($module, /, x, beta, out_dtype=0, out=None, stream=None)\n--\n\n"
     "hbmm_binarize_dense: x fp32 [rows, K] (row stride >= K, unit column stride); returns delta (.) Sign(x) as fp32 or bf16."},
    {"binarize_backward", FAST(py_binarize_backward),
     "binarize_backward($module, /, x, gy, beta, gx=None, stream=None)\n--\n\n"
     "hbmm_binarize_backward: x, gy fp32 [rows, K] (row stride >= K, unit column stride); returns gx = dC/dX."},
    {"connect", py_connect, METH_VARARGS, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding() {
  s_desc = PyUnicode_InternFromString("desc");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  if (!s_desc || !s_cuda_stream) return nullptr;
  PyObject* m = PyModule_Create(&module_def);
  if (m && PyModule_AddStringConstant(m, "BUILT_FOR", HBMM_BUILT_FOR) != 0) Py_CLEAR(m);
  return m;
}
