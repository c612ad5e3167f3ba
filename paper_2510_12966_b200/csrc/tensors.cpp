// Output tensors of the Python binding, several per call. A call that returns per-row outputs makes up to seven of them;
// through torch's Python entry points that takes 12 us, as long as a small verification itself, mostly in parsing
// arguments. Here: 5 us. Every tensor is an allocation of its own, as torch.empty makes it.
#include <ATen/ATen.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/object_ptr.h>

#include <vector>

namespace {

// new_tensors(like, kind, rows, cols, kind, rows, cols, ...): for every triple an uninitialised tensor on the device of the
// tensor `like`: int32 (kind 0) or float32 (kind 1) of shape [rows, cols], or int32 of shape [rows] (kind 2). Returns the
// tensors, then their data pointers.
PyObject* new_tensors(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
  HANDLE_TH_ERRORS
  if (n_args < 1 || n_args % 3 != 1 || !THPVariable_Check(args[0])) {
    PyErr_SetString(PyExc_TypeError, "new_tensors(tensor, kind, rows, cols, ...)");
    return nullptr;
  }
  const Py_ssize_t n = n_args / 3;
  std::vector<int64_t> spec(n_args - 1);
  for (Py_ssize_t i = 1; i < n_args; ++i) {
    spec[i - 1] = PyLong_AsLongLong(args[i]);
    if (spec[i - 1] == -1 && PyErr_Occurred()) return nullptr;
  }
  const auto device = THPVariable_Unpack(args[0]).device();
  std::vector<at::Tensor> made(n);
  {
    pybind11::gil_scoped_release no_gil;
    for (Py_ssize_t i = 0; i < n; ++i) {
      const auto options = at::TensorOptions().device(device).dtype(spec[3 * i] == 1 ? at::kFloat : at::kInt);
      const int64_t shape[2] = {spec[3 * i + 1], spec[3 * i + 2]};
      made[i] = at::empty(at::IntArrayRef(shape, spec[3 * i] == 2 ? 1 : 2), options);
    }
  }
  THPObjectPtr out(PyTuple_New(2 * n));
  if (!out) return nullptr;
  for (Py_ssize_t i = 0; i < n; ++i) {
    PyObject* address = PyLong_FromVoidPtr(made[i].data_ptr());
    if (address == nullptr) return nullptr;
    PyTuple_SET_ITEM(out.get(), n + i, address);
    PyObject* tensor = THPVariable_Wrap(made[i]);
    if (tensor == nullptr) return nullptr;
    PyTuple_SET_ITEM(out.get(), i, tensor);
  }
  return out.release();
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {{"new_tensors", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(new_tensors)), METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_tensors", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__tensors(void) { return PyModule_Create(&module); }
