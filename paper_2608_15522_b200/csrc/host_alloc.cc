// Whole calls for the wrappers of binding.py (below), and for their general way uninitialised tensors: torch.empty without the parsing
// of its Python arguments, which costs twice what the allocation does (2.2 us a tensor; the audio branch's own mask and attention,
// called without buffers, make eight of them in a pass of 40 us).  The same operators through the same dispatcher, caching allocator
// and current stream, and as there without the interpreter lock: an allocation may wait for the GPU.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/ATen.h>
#include <ATen/DimVector.h>
#include <torch/csrc/utils/object_ptr.h>

#include <climits>

#include "../../include/avsa.h"

namespace {

// What `allocate` returns, called without the interpreter lock (which is taken again if it throws, too).
template <typename F>
at::Tensor without_lock(F&& allocate) {
  struct Lock {
    PyThreadState* state = PyEval_SaveThread();
    ~Lock() { PyEval_RestoreThread(state); }
  } lock;
  return allocate();
}

// empty(like, kind, *sizes): kind 0 fp32, 1 int32, 2 uint8, 3 bf16, on the device of `like`
PyObject* py_empty(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  static constexpr at::ScalarType kinds[] = {at::kFloat, at::kInt, at::kByte, at::kBFloat16};
  TORCH_CHECK_TYPE(n >= 2 && n <= 6 && THPVariable_Check(a[0]), "expected a tensor, a kind and up to four sizes");
  const long kind = PyLong_AsLong(a[1]);
  if (kind == -1 && PyErr_Occurred()) return nullptr;
  TORCH_CHECK_VALUE(kind >= 0 && kind < 4, "unknown kind");
  int64_t sizes[4];
  for (Py_ssize_t i = 2; i < n; i++) {
    sizes[i - 2] = PyLong_AsLongLong(a[i]);
    if (sizes[i - 2] == -1 && PyErr_Occurred()) return nullptr;
  }
  const auto options = at::TensorOptions().dtype(kinds[kind]).device(THPVariable_Unpack(a[0]).device());
  return THPVariable_Wrap(without_lock([&] { return at::empty(at::IntArrayRef(sizes, n - 2), options); }));
  END_HANDLE_TH_ERRORS
}

// empty_as(like): bf16 with the shape, strides and device of `like`
PyObject* py_empty_as(PyObject*, PyObject* like) {
  HANDLE_TH_ERRORS
  TORCH_CHECK_TYPE(THPVariable_Check(like), "expected a tensor");
  const at::Tensor& t = THPVariable_Unpack(like);
  const at::DimVector sizes(t.sizes()), strides(t.strides());      // (another thread may change the tensor meanwhile)
  const auto options = at::TensorOptions().dtype(at::kBFloat16).device(t.device());
  return THPVariable_Wrap(without_lock([&] { return at::empty_strided(sizes, strides, options); }));
  END_HANDLE_TH_ERRORS
}

// ------------------------------------------------------------------------------------------------ whole calls
// A wrapper's call in one step for what programs pass: plain tensors on a GPU, ints, floats.  Shapes, strides and pointers are read
// from the tensors themselves instead of through a dozen Python attributes, what the caller did not bring is allocated here, and
// the interpreter lock is free for allocations, workspace query and launches together.  Arguments of another class (a subclass of a tensor,
// an int for a float, no tensor where one has to be), and q, k or v of another type, rank, layout or kind of device, are left to the
// general way with its errors: the function then returns None and has done nothing.  Of the other tensors nothing but the class
// is looked at, as in the general way.  (us: the audio branch's mask and attention without buffers 29.6 -> 21.8; the smallest layer-step,
// three calls with buffers, on the host 21.4 -> 17.0.)

decltype(&avsa_cross_attn_scores) f_cross;
decltype(&avsa_cross_attn_scores_workspace_bytes) f_cross_ws;
decltype(&avsa_build_block_mask) f_mask;
decltype(&avsa_build_block_mask_workspace_bytes) f_mask_ws;
decltype(&avsa_sparse_self_attn) f_sparse;
decltype(&avsa_sparse_self_attn_workspace_bytes) f_sparse_ws;
decltype(&avsa_protected_rows_attn) f_protected;
decltype(&avsa_protected_rows_attn_workspace_bytes) f_protected_ws;
PyObject* o_raw_stream;

// A tensor argument: none, or one held for the length of the call (another thread may drop the caller's).  Another thread may also
// resize it or give it other data: where these are and how many is read once, with the interpreter lock, as are the sizes and
// strides of q, k and v, and nothing is asked of the caller's tensors after that.
struct Arg {
  at::Tensor t;
  void* ptr = nullptr;
  int64_t numel = 0;
  bool there() const { return t.defined(); }
  void read() {
    ptr = t.data_ptr();
    numel = t.numel();
  }
};
bool take(PyObject* o, Arg& a, bool optional) {
  if (o == Py_None) return optional;
  if (!THPVariable_CheckExact(o)) return false;
  a.t = THPVariable_Unpack(o);
  a.read();
  return true;
}
// bf16 [B,H,N,d] on a GPU with a contiguous head dimension
struct View : Arg {
  int64_t size[4], stride[4];
  operator avsa_bf16_4d() const { return avsa_bf16_4d{ptr, stride[0], stride[1], stride[2]}; }
  int dim(int i) const { return static_cast<int>(size[i]); }
};
bool take_view(PyObject* o, View& a) {
  if (!THPVariable_CheckExact(o)) return false;
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.is_cuda() || t.scalar_type() != at::kBFloat16 || t.layout() != at::kStrided || t.dim() != 4 || t.stride(3) != 1) return false;
  a.t = t;
  a.read();
  for (int i = 0; i < 4; i++) {
    a.size[i] = t.size(i);
    a.stride[i] = t.stride(i);
  }
  return true;
}
bool take_int(PyObject* o, int* out) {
  if (!PyLong_CheckExact(o)) return false;
  int overflow;
  const long v = PyLong_AsLongAndOverflow(o, &overflow);
  if (overflow != 0 || v < INT_MIN || v > INT_MAX) return false;
  *out = static_cast<int>(v);
  return true;
}
bool take_float(PyObject* o, float* out) {
  if (!PyFloat_CheckExact(o)) return false;
  *out = static_cast<float>(PyFloat_AS_DOUBLE(o));
  return true;
}
// Where a call runs and what it allocates there: the device of q and its current stream.
struct Place {
  at::Device device;
  void* stream;
  explicit Place(const View& q) : device(q.t.device()), stream(nullptr) {
    THPObjectPtr index(PyLong_FromLong(q.t.get_device()));
    if (!index) throw python_error();
    THPObjectPtr raw(PyObject_CallOneArg(o_raw_stream, index.get()));
    if (!raw) throw python_error();
    stream = PyLong_AsVoidPtr(raw.get());
    if (stream == nullptr && PyErr_Occurred()) throw python_error();
  }
  at::TensorOptions options(at::ScalarType type) const { return at::TensorOptions().dtype(type).device(device); }
  void make(Arg& a, at::ScalarType type, at::IntArrayRef sizes) const {      // what the caller did not bring
    if (a.there()) return;
    a.t = at::empty(sizes, options(type));
    a.read();
  }
  void make_as(Arg& a, const View& like) const {
    if (a.there()) return;
    a.t = at::empty_strided(like.size, like.stride, options(at::kBFloat16));
    a.read();
  }
  void make_ws(Arg& a, size_t bytes) const { make(a, at::kByte, {static_cast<int64_t>(bytes > 256 ? bytes : 256)}); }
};
// The caller's own object where there was one.
PyObject* give(PyObject* given, Arg& a) { return given != Py_None ? Py_NewRef(given) : a.there() ? THPVariable_Wrap(a.t) : Py_NewRef(Py_None); }
template <int N>
PyObject* result(int status, PyObject* (&items)[N]) {
  PyObject* r = PyTuple_New(N + 1);
  PyObject* st = PyLong_FromLong(status);
  bool ok = r != nullptr && st != nullptr;
  for (PyObject* i : items) ok = ok && i != nullptr;
  if (!ok) {
    Py_XDECREF(r);
    Py_XDECREF(st);
    for (PyObject* i : items) Py_XDECREF(i);
    return nullptr;
  }
  PyTuple_SET_ITEM(r, 0, st);
  for (int i = 0; i < N; i++) PyTuple_SET_ITEM(r, i + 1, items[i]);
  return r;
}

// cross(q, k, v, scores, score_beta, score_gamma, softmax_scale, want_o, want_scores, o, lse, ws) -> (status, o, lse, scores, ws)
PyObject* py_cross(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  TORCH_CHECK_TYPE(n == 12 && f_cross != nullptr, "wrong number of arguments, or bind() has not been called");
  View q, k, v;
  Arg scores, o, lse, ws;
  float beta, gamma, scale;
  if (!PyBool_Check(a[7]) || !PyBool_Check(a[8]) || !take_view(a[0], q) || !take_view(a[1], k) || !take_view(a[2], v) ||
      !take(a[8] == Py_True ? a[3] : Py_None, scores, true) || !take_float(a[4], &beta) || !take_float(a[5], &gamma) || !take_float(a[6], &scale) ||
      !take(a[7] == Py_True ? a[9] : Py_None, o, true) || !take(a[10], lse, true) || !take(a[11], ws, true))
    Py_RETURN_NONE;
  const bool want_o = a[7] == Py_True, want_scores = a[8] == Py_True;
  const Place place(q);
  const int B = q.dim(0), H = q.dim(1), Nq = q.dim(2), Nk = k.dim(2), d = q.dim(3);
  int st;
  without_lock([&] {
    if (want_o) place.make_as(o, q);
    place.make(lse, at::kFloat, {B, H, Nq});
    if (want_scores && !scores.there()) {
      place.make(scores, at::kFloat, {B, Nk});
      beta = 0.f;
    }
    if (!ws.there()) place.make_ws(ws, f_cross_ws(B, H, Nq, Nk, d));
    st = f_cross(B, H, Nq, Nk, d, q, k, v, want_o ? o.ptr : nullptr, static_cast<float*>(lse.ptr),
                 want_scores ? static_cast<float*>(scores.ptr) : nullptr, beta, gamma, scale, ws.ptr,
                 static_cast<size_t>(ws.numel), place.stream);
    return at::Tensor();
  });
  PyObject* items[] = {give(a[9], o), give(a[10], lse), give(a[3], scores), give(a[11], ws)};
  return result(st, items);
  END_HANDLE_TH_ERRORS
}

// mask(q, k, scores, n_protect, k_keep, blk, flags, softmax_scale, block_scores, col_idx, col_cnt, prot_tok, prot_blk, ws)
//   -> (status, block_scores, col_idx, col_cnt, prot_tok, prot_blk, ws)
PyObject* py_mask(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  TORCH_CHECK_TYPE(n == 14 && f_mask != nullptr, "wrong number of arguments, or bind() has not been called");
  View q, k;
  Arg scores, bs, idx, cnt, tok, pblk, ws;
  int n_protect, k_keep, blk, flags;
  float scale;
  if (!take_view(a[0], q) || !take_view(a[1], k) || !take(a[2], scores, true) || !take_int(a[3], &n_protect) || !take_int(a[4], &k_keep) ||
      !take_int(a[5], &blk) || blk <= 0 || !take_int(a[6], &flags) || !take_float(a[7], &scale) || !take(a[8], bs, true) ||
      !take(a[9], idx, true) || !take(a[10], cnt, true) || !take(a[11], tok, true) || !take(a[12], pblk, true) || !take(a[13], ws, true))
    Py_RETURN_NONE;
  const Place place(q);
  const int B = q.dim(0), H = q.dim(1), N = q.dim(2), d = q.dim(3);
  const int64_t NB = (static_cast<int64_t>(N) + blk - 1) / blk;
  int st;
  without_lock([&] {
    place.make(bs, at::kFloat, {B, H, NB, NB});
    place.make(idx, at::kInt, {B, H, NB, NB});
    place.make(cnt, at::kInt, {B, H, NB});
    place.make(tok, at::kByte, {B, N});
    place.make(pblk, at::kByte, {B, NB});
    if (!ws.there()) place.make_ws(ws, f_mask_ws(B, H, N, d, blk));
    st = f_mask(B, H, N, d, blk, q, k, static_cast<float*>(scores.ptr), n_protect, k_keep, static_cast<unsigned>(flags), scale,
                static_cast<float*>(bs.ptr), static_cast<int32_t*>(idx.ptr), static_cast<int32_t*>(cnt.ptr),
                static_cast<uint8_t*>(tok.ptr), static_cast<uint8_t*>(pblk.ptr), ws.ptr, static_cast<size_t>(ws.numel), place.stream);
    return at::Tensor();
  });
  PyObject* items[] = {give(a[8], bs), give(a[9], idx), give(a[10], cnt), give(a[11], tok), give(a[12], pblk), give(a[13], ws)};
  return result(st, items);
  END_HANDLE_TH_ERRORS
}

// sparse(q, k, v, col_idx, col_cnt, blk, softmax_scale, want_lse, o, lse, ws) -> (status, o, lse, ws)
PyObject* py_sparse(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  TORCH_CHECK_TYPE(n == 11 && f_sparse != nullptr, "wrong number of arguments, or bind() has not been called");
  View q, k, v;
  Arg idx, cnt, o, lse, ws;
  int blk;
  float scale;
  if (!PyBool_Check(a[7]) || !take_view(a[0], q) || !take_view(a[1], k) || !take_view(a[2], v) || !take(a[3], idx, false) ||
      !take(a[4], cnt, false) || !take_int(a[5], &blk) || !take_float(a[6], &scale) || !take(a[8], o, true) || !take(a[9], lse, true) ||
      !take(a[10], ws, true))
    Py_RETURN_NONE;
  const Place place(q);
  const int B = q.dim(0), H = q.dim(1), N = q.dim(2), d = q.dim(3);
  int st;
  without_lock([&] {
    place.make_as(o, q);
    if (a[7] == Py_True) place.make(lse, at::kFloat, {B, H, N});
    if (!ws.there()) place.make_ws(ws, f_sparse_ws(B, H, N, d, blk));
    st = f_sparse(B, H, N, d, blk, q, k, v, static_cast<int32_t*>(idx.ptr), static_cast<int32_t*>(cnt.ptr), o.ptr,
                  static_cast<float*>(lse.ptr), scale, ws.ptr, static_cast<size_t>(ws.numel), place.stream);
    return at::Tensor();
  });
  PyObject* items[] = {give(a[8], o), give(a[9], lse), give(a[10], ws)};
  return result(st, items);
  END_HANDLE_TH_ERRORS
}

// protected_rows(q, k, v, prot_tok, n_protect, blk, o, lse, softmax_scale, ws) -> (status, ws)
PyObject* py_protected(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  TORCH_CHECK_TYPE(n == 10 && f_protected != nullptr, "wrong number of arguments, or bind() has not been called");
  View q, k, v;
  Arg tok, o, lse, ws;
  int n_protect, blk;
  float scale;
  if (!take_view(a[0], q) || !take_view(a[1], k) || !take_view(a[2], v) || !take(a[3], tok, false) || !take_int(a[4], &n_protect) ||
      !take_int(a[5], &blk) || !take(a[6], o, false) || !take(a[7], lse, true) || !take_float(a[8], &scale) || !take(a[9], ws, true))
    Py_RETURN_NONE;
  const Place place(q);
  const int B = q.dim(0), H = q.dim(1), N = q.dim(2), d = q.dim(3);
  int st;
  without_lock([&] {
    if (!ws.there()) place.make_ws(ws, f_protected_ws(B, H, N, d, blk, n_protect));
    st = f_protected(B, H, N, d, blk, q, k, v, static_cast<uint8_t*>(tok.ptr), n_protect, o.ptr,
                     static_cast<float*>(lse.ptr), scale, ws.ptr, static_cast<size_t>(ws.numel), place.stream);
    return at::Tensor();
  });
  PyObject* items[] = {give(a[9], ws)};
  return result(st, items);
  END_HANDLE_TH_ERRORS
}

// bind(addresses of cross, mask, sparse, protected rows and of their workspace queries, reader of the raw current stream)
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  TORCH_CHECK_TYPE(n == 9, "wrong number of arguments");
  void* p[8];
  for (int i = 0; i < 8; i++) {
    p[i] = PyLong_AsVoidPtr(a[i]);
    if (p[i] == nullptr) {
      TORCH_CHECK_VALUE(PyErr_Occurred(), "a null address");
      return nullptr;
    }
  }
  o_raw_stream = Py_NewRef(a[8]);
  f_cross = reinterpret_cast<decltype(f_cross)>(p[0]);
  f_mask = reinterpret_cast<decltype(f_mask)>(p[1]);
  f_sparse = reinterpret_cast<decltype(f_sparse)>(p[2]);
  f_protected = reinterpret_cast<decltype(f_protected)>(p[3]);
  f_cross_ws = reinterpret_cast<decltype(f_cross_ws)>(p[4]);
  f_mask_ws = reinterpret_cast<decltype(f_mask_ws)>(p[5]);
  f_sparse_ws = reinterpret_cast<decltype(f_sparse_ws)>(p[6]);
  f_protected_ws = reinterpret_cast<decltype(f_protected_ws)>(p[7]);
  Py_RETURN_NONE;
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"empty", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_empty)), METH_FASTCALL, nullptr},
    {"empty_as", py_empty_as, METH_O, nullptr},
    {"bind", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_bind)), METH_FASTCALL, nullptr},
    {"cross", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_cross)), METH_FASTCALL, nullptr},
    {"mask", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_mask)), METH_FASTCALL, nullptr},
    {"sparse", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_sparse)), METH_FASTCALL, nullptr},
    {"protected_rows", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_protected)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_avsa_alloc", "uninitialised tensors and whole calls for the wrappers", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" __attribute__((visibility("default"))) PyObject* PyInit__avsa_alloc(void) { return PyModule_Create(&module); }
