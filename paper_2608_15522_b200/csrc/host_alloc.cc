// Uninitialised tensors for the wrappers of binding.py: torch.empty without the parsing of its Python arguments, which costs
// twice what the allocation does (2.2 us a tensor; the audio branch's own mask and attention, called without buffers, make
// eight of them in a pass of 40 us).  The same operators through the same dispatcher, caching allocator and current stream, and
// as there without the interpreter lock: an allocation may wait for the GPU.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <ATen/ATen.h>
#include <ATen/DimVector.h>

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

PyMethodDef methods[] = {
    {"empty", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(py_empty)), METH_FASTCALL, nullptr},
    {"empty_as", py_empty_as, METH_O, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_avsa_alloc", "uninitialised tensors", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

extern "C" __attribute__((visibility("default"))) PyObject* PyInit__avsa_alloc(void) { return PyModule_Create(&module); }
