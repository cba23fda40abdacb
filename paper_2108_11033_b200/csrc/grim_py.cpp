// The calls of the binding that run once per product, as a CPython extension: arguments are read straight from the
// torch tensors (no per-call ctypes structures, no attribute look-ups in Python) and handed to the C ABI of libgrim.
// A small product's kernel takes a few microseconds, so what the host spends per call is what such a call costs:
// 19 us through ctypes, about 6 us through this file (256 x 256 weight, 64 columns).
//
// Marshalling only, with the checks and exceptions of the Python binding: AssertionError for a tensor that is not on
// the GPU or not laid out as the call needs it, TypeError for an unsupported data type, GrimError for a status.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstring>

#include "grim.h"

namespace {

PyObject* g_error_class = nullptr;  // binding.GrimError

// Argument list of one call: positional and keyword arguments matched to `names`, borrowed references, null = not given.
constexpr int kMaxArgs = 10;
struct Args {
  PyObject* v[kMaxArgs] = {};
};

bool parse(const char* fn, const char* const* names, int n, int required, PyObject* const* args, Py_ssize_t nargs,
           PyObject* kwnames, Args& out) {
  if (nargs > n) {
    PyErr_Format(PyExc_TypeError, "%s() takes at most %d arguments (%zd given)", fn, n, nargs);
    return false;
  }
  for (Py_ssize_t i = 0; i < nargs; ++i) out.v[i] = args[i];
  const Py_ssize_t nk = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
  for (Py_ssize_t k = 0; k < nk; ++k) {
    const char* key = PyUnicode_AsUTF8(PyTuple_GET_ITEM(kwnames, k));
    int at = -1;
    for (int i = 0; key && i < n; ++i)
      if (std::strcmp(key, names[i]) == 0) at = i;
    if (at < 0 || out.v[at]) {
      PyErr_Format(PyExc_TypeError, at < 0 ? "%s() got an unexpected keyword argument '%s'" : "%s() got multiple values for argument '%s'",
                   fn, key ? key : "?");
      return false;
    }
    out.v[at] = args[nargs + k];
  }
  for (int i = 0; i < required; ++i)
    if (!out.v[i]) {
      PyErr_Format(PyExc_TypeError, "%s() missing required argument '%s'", fn, names[i]);
      return false;
    }
  return true;
}

// The integer that grim_bcr_pack and grim_gru_create return, None, or a ctypes.c_void_p.
bool to_handle(PyObject* o, void** out) {
  PyObject* value = !PyLong_Check(o) && o != Py_None && PyObject_HasAttrString(o, "value") ? PyObject_GetAttrString(o, "value") : nullptr;
  if (value) o = value;
  *out = o == Py_None ? nullptr : PyLong_AsVoidPtr(o);
  Py_XDECREF(value);
  return !(*out == nullptr && PyErr_Occurred());
}

bool to_int(PyObject* o, int dflt, int* out) {
  if (!o) { *out = dflt; return true; }
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) return false;
  *out = (int)v;
  return true;
}

const at::Tensor* to_tensor(const char* fn, PyObject* o) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "%s(): expected a torch tensor, got %s", fn, Py_TYPE(o)->tp_name);
    return nullptr;
  }
  return &THPVariable_Unpack(o);
}

bool to_dtype(const at::Tensor& t, grim_dtype_t* out) {
  if (t.scalar_type() == at::kFloat) { *out = GRIM_F32; return true; }
  if (t.scalar_type() == at::kBFloat16) { *out = GRIM_BF16; return true; }
  PyErr_Format(PyExc_TypeError, "unsupported tensor dtype %s", c10::toString(t.scalar_type()));
  return false;
}

bool fail(const char* fn, const char* what) {
  PyErr_Format(PyExc_AssertionError, "%s(): %s", fn, what);
  return false;
}

// A vector counts as a matrix of one column.
bool to_mat(const char* fn, PyObject* o, grim_mat_t* m) {
  const at::Tensor* t = to_tensor(fn, o);
  if (!t) return false;
  const int64_t dim = t->dim();
  if (!t->is_cuda() || dim < 1 || dim > 2 || (dim == 2 && t->stride(1) != 1))
    return fail(fn, "operands are CUDA matrices whose rows are contiguous");
  m->rows = t->size(0);
  m->cols = dim == 2 ? t->size(1) : 1;
  m->ld = t->stride(0);
  if (m->rows <= 1 && m->ld < m->cols) m->ld = m->cols;
  m->ptr = t->data_ptr();
  return to_dtype(*t, &m->dtype);
}

bool to_contiguous(const char* fn, PyObject* o, const at::Tensor** out) {
  const at::Tensor* t = to_tensor(fn, o);
  if (!t) return false;
  if (!t->is_cuda() || !t->is_contiguous()) return fail(fn, "operands are contiguous CUDA tensors");
  *out = t;
  return true;
}

// Pointer of an optional tensor.
bool to_opt_ptr(const char* fn, PyObject* o, void** out) {
  *out = nullptr;
  if (!o || o == Py_None) return true;
  const at::Tensor* t = to_tensor(fn, o);
  if (!t) return false;
  *out = t->data_ptr();
  return true;
}

// None: torch's current stream; an object with a cuda_stream attribute; or the stream's address, as anything int() takes.
bool to_stream(PyObject* o, grim_stream_t* out) {
  if (!o || o == Py_None) {
    *out = (grim_stream_t)c10::cuda::getCurrentCUDAStream().stream();
    return true;
  }
  void* p = nullptr;
  if (PyLong_Check(o)) {
    p = PyLong_AsVoidPtr(o);
  } else {
    PyObject* number = PyObject_HasAttrString(o, "cuda_stream") ? PyObject_GetAttrString(o, "cuda_stream") : PyNumber_Long(o);
    if (!number) return false;
    p = PyLong_AsVoidPtr(number);
    Py_DECREF(number);
  }
  if (!p && PyErr_Occurred()) return false;
  *out = (grim_stream_t)p;
  return true;
}

PyObject* finish(grim_status_t st, const char* where) {
  if (st == GRIM_OK) Py_RETURN_NONE;
  if (!g_error_class) {
    PyErr_Format(PyExc_RuntimeError, "%s: %s (status %d)", where, grim_status_string(st), (int)st);
    return nullptr;
  }
  PyObject* e = PyObject_CallFunction(g_error_class, "is", (int)st, where);
  if (e) {
    PyErr_SetObject(g_error_class, e);
    Py_DECREF(e);
  }
  return nullptr;
}

// Runs `call` without the interpreter lock (a launch may block when the queue is full).
template <typename F>
PyObject* run(const char* where, F call) {
  grim_status_t st;
  Py_BEGIN_ALLOW_THREADS
  st = call();
  Py_END_ALLOW_THREADS
  return finish(st, where);
}

// C++ exceptions (torch raises them, e.g. without a GPU) become RuntimeError.
template <typename F>
PyObject* guarded(F body) {
  try {
    return body();
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

#define GRIM_PARSE(fn, required, ...)                                                                             \
  static const char* const names[] = {__VA_ARGS__};                                                               \
  static_assert(sizeof(names) / sizeof(names[0]) <= kMaxArgs, "");                                                \
  Args a;                                                                                                         \
  const char* const where = fn;                                                                                   \
  if (!parse(fn, names, (int)(sizeof(names) / sizeof(names[0])), required, args, nargs, kwnames, a)) return nullptr

using Vec = PyObject* const*;

PyObject* py_spmm(PyObject*, Vec args, Py_ssize_t nargs, PyObject* kwnames) {
  return guarded([&]() -> PyObject* {
    GRIM_PARSE("grim_bcr_spmm", 3, "h", "X", "Y", "stream");
    void* h;
    grim_mat_t x, y;
    grim_stream_t s;
    if (!to_handle(a.v[0], &h) || !to_mat(where, a.v[1], &x) || !to_mat(where, a.v[2], &y) || !to_stream(a.v[3], &s)) return nullptr;
    return run(where, [&] { return grim_bcr_spmm((grim_bcr_t)h, &x, &y, s); });
  });
}

PyObject* py_spmm_ex(PyObject*, Vec args, Py_ssize_t nargs, PyObject* kwnames) {
  return guarded([&]() -> PyObject* {
    GRIM_PARSE("grim_bcr_spmm_ex", 3, "h", "X", "Y", "tile_n", "path", "stream");
    void* h;
    grim_mat_t x, y;
    grim_stream_t s;
    grim_tune_t tune = {};
    if (!to_handle(a.v[0], &h) || !to_mat(where, a.v[1], &x) || !to_mat(where, a.v[2], &y) || !to_int(a.v[3], 0, &tune.tile_n) ||
        !to_int(a.v[4], 0, &tune.path) || !to_stream(a.v[5], &s))
      return nullptr;
    return run(where, [&] { return grim_bcr_spmm_ex((grim_bcr_t)h, &x, &y, &tune, s); });
  });
}

PyObject* py_conv2d(PyObject*, Vec args, Py_ssize_t nargs, PyObject* kwnames) {
  return guarded([&]() -> PyObject* {
    GRIM_PARSE("grim_bcr_conv2d", 4, "h", "x", "out", "ksize", "stride", "pad", "bias", "relu", "stream", "kernel_flags");
    void *h, *bias;
    const at::Tensor *x, *out;
    grim_stream_t s;
    int ksize, kernel_flags;
    grim_conv_desc_t d = {};
    if (!to_handle(a.v[0], &h) || !to_contiguous(where, a.v[1], &x) || !to_contiguous(where, a.v[2], &out) ||
        !to_int(a.v[3], 0, &ksize) || !to_int(a.v[4], 1, &d.stride) || !to_int(a.v[5], 0, &d.pad) || !to_opt_ptr(where, a.v[6], &bias) ||
        !to_stream(a.v[8], &s) || !to_int(a.v[9], 0, &kernel_flags) || !to_dtype(*x, &d.in_dtype) || !to_dtype(*out, &d.out_dtype))
      return nullptr;
    if (x->dim() != 4) { fail(where, "the input has four dimensions"); return nullptr; }
    const int relu = a.v[7] ? PyObject_IsTrue(a.v[7]) : 0;
    if (relu < 0) return nullptr;
    d.N = x->size(0); d.C = x->size(1); d.H = x->size(2); d.W = x->size(3);
    d.KH = d.KW = ksize;
    d.bias_dev = static_cast<const float*>(bias);
    d.flags = (relu ? GRIM_CONV_RELU : 0u) | (uint32_t)kernel_flags;
    const void* in = x->data_ptr();
    void* o = out->data_ptr();
    return run(where, [&] { return grim_bcr_conv2d((grim_bcr_t)h, &d, in, o, s); });
  });
}

PyObject* py_maxpool(PyObject*, Vec args, Py_ssize_t nargs, PyObject* kwnames) {
  return guarded([&]() -> PyObject* {
    GRIM_PARSE("grim_maxpool2x2", 2, "x", "out", "stream");
    const at::Tensor *x, *out;
    grim_stream_t s;
    grim_dtype_t dt;
    if (!to_contiguous(where, a.v[0], &x) || !to_contiguous(where, a.v[1], &out) || !to_stream(a.v[2], &s) || !to_dtype(*x, &dt)) return nullptr;
    if (x->dim() != 4) { PyErr_SetString(PyExc_ValueError, "grim_maxpool2x2(): the input has four dimensions"); return nullptr; }
    const void* in = x->data_ptr();
    void* o = out->data_ptr();
    const int64_t n = x->size(0), c = x->size(1), hh = x->size(2), ww = x->size(3);
    return run(where, [&] { return grim_maxpool2x2(in, o, n, c, hh, ww, dt, s); });
  });
}

using SeqFn = grim_status_t (*)(grim_gru_t, const float*, int64_t, const float*, float*, float*, grim_stream_t);
PyObject* gru_seq(const char* fn, SeqFn call, Vec args, Py_ssize_t nargs, PyObject* kwnames) {
  return guarded([&]() -> PyObject* {
    GRIM_PARSE(fn, 3, "g", "x", "y", "h0", "hT", "stream");
    void *g, *h0, *hT;
    const at::Tensor *x, *y;
    grim_stream_t s;
    if (!to_handle(a.v[0], &g) || !to_contiguous(where, a.v[1], &x) || !to_contiguous(where, a.v[2], &y) ||
        !to_opt_ptr(where, a.v[3], &h0) || !to_opt_ptr(where, a.v[4], &hT) || !to_stream(a.v[5], &s))
      return nullptr;
    const float* xp = static_cast<const float*>(x->data_ptr());
    float* yp = static_cast<float*>(y->data_ptr());
    const int64_t T = x->size(0);
    return run(where, [&] { return call((grim_gru_t)g, xp, T, static_cast<const float*>(h0), yp, static_cast<float*>(hT), s); });
  });
}
PyObject* py_gru_seq(PyObject*, Vec args, Py_ssize_t nargs, PyObject* kwnames) {
  return gru_seq("grim_gru_seq", grim_gru_seq, args, nargs, kwnames);
}
PyObject* py_gru_seq_static(PyObject*, Vec args, Py_ssize_t nargs, PyObject* kwnames) {
  return gru_seq("grim_gru_seq_static", grim_gru_seq_static, args, nargs, kwnames);
}

PyObject* py_gru_step(PyObject*, Vec args, Py_ssize_t nargs, PyObject* kwnames) {
  return guarded([&]() -> PyObject* {
    GRIM_PARSE("grim_gru_step", 3, "g", "x", "h", "y", "stream");
    void *g, *y;
    const at::Tensor *x, *h;
    grim_stream_t s;
    if (!to_handle(a.v[0], &g) || !to_contiguous(where, a.v[1], &x) || !to_contiguous(where, a.v[2], &h) ||
        !to_opt_ptr(where, a.v[3], &y) || !to_stream(a.v[4], &s))
      return nullptr;
    if (x->dim() != 2 || h->dim() != 3) { fail(where, "x has two dimensions and h three"); return nullptr; }
    const float* xp = static_cast<const float*>(x->data_ptr());
    float* hp = static_cast<float*>(h->data_ptr());
    const int64_t B = x->size(0);
    return run(where, [&] { return grim_gru_step((grim_gru_t)g, xp, B, hp, static_cast<float*>(y), s); });
  });
}

PyObject* py_set_error_class(PyObject*, PyObject* cls) {
  Py_XINCREF(cls);
  Py_XDECREF(g_error_class);
  g_error_class = cls;
  Py_RETURN_NONE;
}

#define GRIM_METHOD(name, fn, doc) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(fn)), METH_FASTCALL | METH_KEYWORDS, doc}
PyMethodDef methods[] = {
    GRIM_METHOD("grim_bcr_spmm", py_spmm, "grim_bcr_spmm(h, X, Y, stream=None)"),
    GRIM_METHOD("grim_bcr_spmm_ex", py_spmm_ex, "grim_bcr_spmm_ex(h, X, Y, tile_n=0, path=0, stream=None)"),
    GRIM_METHOD("grim_bcr_conv2d", py_conv2d,
                "grim_bcr_conv2d(h, x, out, ksize, stride=1, pad=0, bias=None, relu=False, stream=None, kernel_flags=0)"),
    GRIM_METHOD("grim_maxpool2x2", py_maxpool, "grim_maxpool2x2(x, out, stream=None)"),
    GRIM_METHOD("grim_gru_seq", py_gru_seq, "grim_gru_seq(g, x, y, h0=None, hT=None, stream=None)"),
    GRIM_METHOD("grim_gru_seq_static", py_gru_seq_static,
                "grim_gru_seq_static(g, x, y, h0=None, hT=None, stream=None)\n\ngrim_gru_seq for callers that may not allocate device "
                "memory: scratch comes from a fixed 8 MiB array inside the library (shared by all calls; see include/grim.h for the size limit)."),
    GRIM_METHOD("grim_gru_step", py_gru_step, "grim_gru_step(g, x, h, y=None, stream=None)"),
    {"set_error_class", py_set_error_class, METH_O, "set_error_class(cls): the exception raised for a status other than GRIM_OK"},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_grim_py", "Per-product calls of libgrim on torch tensors.", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__grim_py() { return PyModule_Create(&module); }
