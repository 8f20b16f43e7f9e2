// Argument marshalling between Python tensors and the C ABI of libavsa.so, as a CPython extension.
// The same marshalling through ctypes (a structure per tensor, a stream object, twenty converted arguments) took 10 us
// of every call, as much as the launches themselves: a layer-step of 256 tokens was three calls of 20-26 us on the
// host against 31 us of work on the device.  Here it is attribute reads and one C call, with the interpreter lock
// released around it.  The tensors' allocation and the defaults stay in binding.py; the checks are the ones made there
// before (a ValueError for a tensor that the library could not describe, everything else a status of the library).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "../../include/avsa.h"

namespace {

// entry points of the library that binding.py has loaded, torch.bfloat16 and the reader of the current stream
decltype(&avsa_cross_attn_scores) f_cross;
decltype(&avsa_build_block_mask) f_mask;
decltype(&avsa_sparse_self_attn) f_sparse;
decltype(&avsa_protected_rows_attn) f_protected;
decltype(&avsa_cache_indicators) f_indicators;
PyObject *o_bfloat16, *o_raw_stream;
PyObject *s_dtype, *s_is_cuda, *s_shape, *s_stride, *s_data_ptr, *s_numel, *s_get_device, *s_is_contiguous;

// Reads fail by setting the Python error; `ok` carries that through a call's argument list.
bool read_ptr(PyObject* t, void** out) {
  *out = nullptr;
  if (t == Py_None) return true;
  PyObject* r = PyObject_CallMethodNoArgs(t, s_data_ptr);
  if (r == nullptr) return false;
  *out = PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return !PyErr_Occurred();
}
bool read_int(PyObject* v, int* out) {
  PyObject* n = PyNumber_Long(v);
  if (n == nullptr) return false;
  *out = static_cast<int>(PyLong_AsUnsignedLongMask(n));
  Py_DECREF(n);
  return !PyErr_Occurred();
}
// an argument that binding.py does not convert: only an int, as a C prototype would have it (block size 64.9 is not 64)
bool read_strict_int(PyObject* v, int* out) {
  if (PyLong_Check(v)) return read_int(v, out);
  PyErr_Format(PyExc_TypeError, "expected an int, got %s", Py_TYPE(v)->tp_name);
  return false;
}
bool read_float(PyObject* v, float* out) {
  PyObject* f = PyNumber_Float(v);
  if (f == nullptr) return false;
  *out = static_cast<float>(PyFloat_AS_DOUBLE(f));
  Py_DECREF(f);
  return true;
}
bool read_numel(PyObject* t, size_t* out) {
  PyObject* r = PyObject_CallMethodNoArgs(t, s_numel);
  if (r == nullptr) return false;
  *out = PyLong_AsSize_t(r);
  Py_DECREF(r);
  return !PyErr_Occurred();
}
bool attr_is(PyObject* t, PyObject* name, PyObject* want, bool* same) {
  PyObject* r = PyObject_GetAttr(t, name);
  if (r == nullptr) return false;
  *same = r == want;
  Py_DECREF(r);
  return true;
}
bool read_tuple(PyObject* tuple, int64_t* out, Py_ssize_t n) {      // steals the reference
  if (tuple == nullptr) return false;
  bool ok = PyTuple_Check(tuple) && PyTuple_GET_SIZE(tuple) == n;
  if (!ok) PyErr_Format(PyExc_ValueError, "expected a tensor of %zd dimensions", n);
  for (Py_ssize_t i = 0; ok && i < n; i++) {
    out[i] = PyLong_AsLongLong(PyTuple_GET_ITEM(tuple, i));
    if (out[i] == -1 && PyErr_Occurred()) ok = false;
  }
  Py_DECREF(tuple);
  return ok;
}
bool read_shape(PyObject* t, int64_t* shape, Py_ssize_t n) { return read_tuple(PyObject_GetAttr(t, s_shape), shape, n); }
// one extent of a tensor of any rank
bool read_extent(PyObject* t, Py_ssize_t axis, int64_t* out) {
  PyObject* shape = PyObject_GetAttr(t, s_shape);
  if (shape == nullptr) return false;
  PyObject* v = PySequence_GetItem(shape, axis);
  Py_DECREF(shape);
  if (v == nullptr) return false;
  *out = PyLong_AsLongLong(v);
  Py_DECREF(v);
  return !PyErr_Occurred();
}

// bf16 [B,H,N,d] on a CUDA device with a contiguous head dimension
bool read_view(PyObject* t, avsa_bf16_4d* out) {
  bool bf16, cuda;
  if (!attr_is(t, s_dtype, o_bfloat16, &bf16) || !attr_is(t, s_is_cuda, Py_True, &cuda)) return false;
  PyObject* strides = PyObject_CallMethodNoArgs(t, s_stride);
  if (strides == nullptr) return false;
  if (!bf16 || !cuda || !PyTuple_Check(strides) || PyTuple_GET_SIZE(strides) != 4) {
    Py_DECREF(strides);
    PyErr_SetString(PyExc_ValueError, "expected a CUDA bf16 tensor [B,H,N,d]");
    return false;
  }
  int64_t st[4];
  if (!read_tuple(strides, st, 4)) return false;
  if (st[3] != 1) {
    PyErr_SetString(PyExc_ValueError, "the head dimension must be contiguous");
    return false;
  }
  void* p;
  if (!read_ptr(t, &p)) return false;
  *out = avsa_bf16_4d{p, st[0], st[1], st[2]};
  return true;
}
bool read_optional_view(PyObject* t, avsa_bf16_4d* out) {      // None is the null view
  *out = avsa_bf16_4d{nullptr, 0, 0, 0};
  return t == Py_None || read_view(t, out);
}
// current stream of the tensor's device (a tensor in host memory has none: its index is -1, which the reader of the
// stream would take for the current device)
bool read_stream(PyObject* t, void** out) {
  PyObject* dev = PyObject_CallMethodNoArgs(t, s_get_device);
  if (dev == nullptr) return false;
  const long index = PyLong_AsLong(dev);
  if (index < 0) {
    Py_DECREF(dev);
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "expected a tensor on a CUDA device");
    return false;
  }
  PyObject* r = PyObject_CallOneArg(o_raw_stream, dev);
  Py_DECREF(dev);
  if (r == nullptr) return false;
  *out = PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return !PyErr_Occurred();
}
bool arity(Py_ssize_t got, Py_ssize_t want) {
  if (got == want && f_cross != nullptr) return true;
  PyErr_SetString(PyExc_TypeError, f_cross == nullptr ? "bind() has not been called" : "wrong number of arguments");
  return false;
}

// bind(addresses of the five entry points, torch.bfloat16, reader of the raw current stream)
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 7) {
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
    return nullptr;
  }
  void* p[5];
  for (int i = 0; i < 5; i++) {
    p[i] = PyLong_AsVoidPtr(a[i]);
    if (PyErr_Occurred()) return nullptr;
  }
  o_bfloat16 = Py_NewRef(a[5]);
  o_raw_stream = Py_NewRef(a[6]);
  f_mask = reinterpret_cast<decltype(f_mask)>(p[1]);
  f_sparse = reinterpret_cast<decltype(f_sparse)>(p[2]);
  f_protected = reinterpret_cast<decltype(f_protected)>(p[3]);
  f_indicators = reinterpret_cast<decltype(f_indicators)>(p[4]);
  f_cross = reinterpret_cast<decltype(f_cross)>(p[0]);
  Py_RETURN_NONE;
}

// cross(q, k, v, o, lse, scores, beta, gamma, softmax_scale, ws) -> status
PyObject* py_cross(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!arity(n, 10)) return nullptr;
  int64_t qs[4], ks[4];
  avsa_bf16_4d q, k, v;
  void *o, *lse, *scores, *ws, *stream;
  float beta, gamma, scale;
  size_t ws_bytes;
  if (!read_shape(a[0], qs, 4) || !read_shape(a[1], ks, 4) || !read_view(a[0], &q) || !read_view(a[1], &k) ||
      !read_view(a[2], &v) || !read_ptr(a[3], &o) || !read_ptr(a[4], &lse) || !read_ptr(a[5], &scores) ||
      !read_float(a[6], &beta) || !read_float(a[7], &gamma) || !read_float(a[8], &scale) || !read_ptr(a[9], &ws) ||
      !read_numel(a[9], &ws_bytes) || !read_stream(a[0], &stream))
    return nullptr;
  int st;
  Py_BEGIN_ALLOW_THREADS;
  st = f_cross(static_cast<int>(qs[0]), static_cast<int>(qs[1]), static_cast<int>(qs[2]), static_cast<int>(ks[2]),
               static_cast<int>(qs[3]), q, k, v, o, static_cast<float*>(lse), static_cast<float*>(scores), beta, gamma, scale,
               ws, ws_bytes, stream);
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(st);
}

// mask((B, H, N, d), blk, q, k, scores, n_protect, k_keep, flags, softmax_scale, block_scores, col_idx, col_cnt,
//      prot_tok, prot_blk, ws) -> status
PyObject* py_mask(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!arity(n, 15)) return nullptr;
  int64_t sh[4];
  avsa_bf16_4d q, k;
  void *scores, *bs, *idx, *cnt, *tok, *pblk, *ws, *stream;
  int blk, n_protect, k_keep, flags;
  float scale;
  size_t ws_bytes;
  if (!read_tuple(Py_NewRef(a[0]), sh, 4) || !read_strict_int(a[1], &blk) || !read_optional_view(a[2], &q) ||
      !read_optional_view(a[3], &k) || !read_ptr(a[4], &scores) || !read_int(a[5], &n_protect) || !read_int(a[6], &k_keep) || !read_int(a[7], &flags) ||
      !read_float(a[8], &scale) || !read_ptr(a[9], &bs) || !read_ptr(a[10], &idx) || !read_ptr(a[11], &cnt) ||
      !read_ptr(a[12], &tok) || !read_ptr(a[13], &pblk) || !read_ptr(a[14], &ws) || !read_numel(a[14], &ws_bytes) ||
      !read_stream(a[2] != Py_None ? a[2] : a[9], &stream))
    return nullptr;
  int st;
  Py_BEGIN_ALLOW_THREADS;
  st = f_mask(static_cast<int>(sh[0]), static_cast<int>(sh[1]), static_cast<int>(sh[2]), static_cast<int>(sh[3]), blk, q, k,
              static_cast<float*>(scores), n_protect, k_keep, static_cast<unsigned>(flags), scale, static_cast<float*>(bs),
              static_cast<int32_t*>(idx), static_cast<int32_t*>(cnt), static_cast<uint8_t*>(tok), static_cast<uint8_t*>(pblk),
              ws, ws_bytes, stream);
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(st);
}

// sparse(q, k, v, col_idx, col_cnt, blk, o, lse, softmax_scale, ws) -> status
PyObject* py_sparse(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!arity(n, 10)) return nullptr;
  int64_t sh[4];
  avsa_bf16_4d q, k, v;
  void *idx, *cnt, *o, *lse, *ws, *stream;
  int blk;
  float scale;
  size_t ws_bytes;
  if (!read_shape(a[0], sh, 4) || !read_view(a[0], &q) || !read_view(a[1], &k) || !read_view(a[2], &v) ||
      !read_ptr(a[3], &idx) || !read_ptr(a[4], &cnt) || !read_strict_int(a[5], &blk) || !read_ptr(a[6], &o) ||
      !read_ptr(a[7], &lse) || !read_float(a[8], &scale) || !read_ptr(a[9], &ws) || !read_numel(a[9], &ws_bytes) ||
      !read_stream(a[0], &stream))
    return nullptr;
  int st;
  Py_BEGIN_ALLOW_THREADS;
  st = f_sparse(static_cast<int>(sh[0]), static_cast<int>(sh[1]), static_cast<int>(sh[2]), static_cast<int>(sh[3]), blk, q, k,
                v, static_cast<int32_t*>(idx), static_cast<int32_t*>(cnt), o, static_cast<float*>(lse), scale, ws, ws_bytes,
                stream);
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(st);
}

// protected_rows(q, k, v, prot_tok, n_protect, blk, o, lse, softmax_scale, ws) -> status
PyObject* py_protected(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!arity(n, 10)) return nullptr;
  int64_t sh[4];
  avsa_bf16_4d q, k, v;
  void *tok, *o, *lse, *ws, *stream;
  int n_protect, blk;
  float scale;
  size_t ws_bytes;
  if (!read_shape(a[0], sh, 4) || !read_view(a[0], &q) || !read_view(a[1], &k) || !read_view(a[2], &v) ||
      !read_ptr(a[3], &tok) || !read_int(a[4], &n_protect) || !read_strict_int(a[5], &blk) || !read_ptr(a[6], &o) ||
      !read_ptr(a[7], &lse) || !read_float(a[8], &scale) || !read_ptr(a[9], &ws) || !read_numel(a[9], &ws_bytes) ||
      !read_stream(a[0], &stream))
    return nullptr;
  int st;
  Py_BEGIN_ALLOW_THREADS;
  st = f_protected(static_cast<int>(sh[0]), static_cast<int>(sh[1]), static_cast<int>(sh[2]), static_cast<int>(sh[3]), blk, q,
                   k, v, static_cast<uint8_t*>(tok), n_protect, o, static_cast<float*>(lse), scale, ws, ws_bytes, stream);
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(st);
}

// indicators(y_v, yhat_v, y_a, yhat_a, prot_tok, s_cur, s_anchor, lambda_p, lambda_s, tau, eps, out, ws) -> status
PyObject* py_indicators(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!arity(n, 13)) return nullptr;
  int64_t vs[3], na;
  void *y[4], *tok, *cur, *anchor, *out, *ws, *stream;
  float lp, ls, tau, eps;
  size_t ws_bytes;
  for (int i = 0; i < 4; i++) {
    bool bf16, cuda;
    if (!attr_is(a[i], s_dtype, o_bfloat16, &bf16) || !attr_is(a[i], s_is_cuda, Py_True, &cuda)) return nullptr;
    PyObject* c = PyObject_CallMethodNoArgs(a[i], s_is_contiguous);
    if (c == nullptr) return nullptr;
    const bool contiguous = c == Py_True;
    Py_DECREF(c);
    if (!bf16 || !cuda || !contiguous) {
      PyErr_SetString(PyExc_ValueError, "expected contiguous CUDA bf16 tensors");
      return nullptr;
    }
    if (!read_ptr(a[i], &y[i])) return nullptr;
  }
  if (!read_shape(a[0], vs, 3) || !read_extent(a[2], 1, &na) || !read_ptr(a[4], &tok) || !read_ptr(a[5], &cur) ||
      !read_ptr(a[6], &anchor) || !read_float(a[7], &lp) || !read_float(a[8], &ls) || !read_float(a[9], &tau) ||
      !read_float(a[10], &eps) || !read_ptr(a[11], &out) || !read_ptr(a[12], &ws) || !read_numel(a[12], &ws_bytes) ||
      !read_stream(a[0], &stream))
    return nullptr;
  int st;
  Py_BEGIN_ALLOW_THREADS;
  st = f_indicators(static_cast<int>(vs[0]), static_cast<int>(vs[1]), static_cast<int>(na), static_cast<int>(vs[2]), y[0],
                    y[1], y[2], y[3], static_cast<uint8_t*>(tok), static_cast<float*>(cur), static_cast<float*>(anchor), lp, ls,
                    tau, eps, static_cast<float*>(out), ws, ws_bytes, stream);
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(st);
}

PyMethodDef methods[] = {
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_bind)), METH_FASTCALL, nullptr},
    {"cross", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_cross)), METH_FASTCALL, nullptr},
    {"mask", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_mask)), METH_FASTCALL, nullptr},
    {"sparse", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_sparse)), METH_FASTCALL, nullptr},
    {"protected_rows", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_protected)), METH_FASTCALL, nullptr},
    {"indicators", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_indicators)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_avsa_host", "argument marshalling for libavsa.so", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" __attribute__((visibility("default"))) PyObject* PyInit__avsa_host(void) {
  struct { PyObject** s; const char* text; } names[] = {
      {&s_dtype, "dtype"}, {&s_is_cuda, "is_cuda"}, {&s_shape, "shape"}, {&s_stride, "stride"}, {&s_data_ptr, "data_ptr"},
      {&s_numel, "numel"}, {&s_get_device, "get_device"}, {&s_is_contiguous, "is_contiguous"}};
  for (auto& e : names) {
    *e.s = PyUnicode_InternFromString(e.text);
    if (*e.s == nullptr) return nullptr;
  }
  return PyModule_Create(&module);
}
