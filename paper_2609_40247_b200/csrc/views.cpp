// Tensors over memory the library owns, made without the interpreter's indexing machinery: a
// result has up to nineteen columns, and taking a slice of a tensor from Python costs 1.4 us (here
// 0.2), wrapping an address through __cuda_array_interface__ eight.
#include <Python.h>

#include <ATen/ops/from_blob.h>
#include <torch/csrc/autograd/python_variable.h>

// wrap(address, nbytes, device index, owner): uint8 tensor that keeps `owner` alive
static PyObject *wrap(PyObject *, PyObject *const *args, Py_ssize_t n) {
  if (n != 4) {
    PyErr_SetString(PyExc_TypeError, "wrap(address, nbytes, device, owner)");
    return nullptr;
  }
  void *p = PyLong_AsVoidPtr(args[0]);
  const long long bytes = PyLong_AsLongLong(args[1]), dev = PyLong_AsLongLong(args[2]);
  if (PyErr_Occurred()) return nullptr;
  PyObject *owner = args[3];
  try {
    const at::Device device(at::kCUDA, (c10::DeviceIndex)dev);
    Py_INCREF(owner);
    at::Tensor t = at::for_blob(p, {(int64_t)bytes})
                       .deleter([owner](void *) {
                         if (!Py_IsInitialized()) return;
                         const PyGILState_STATE g = PyGILState_Ensure();
                         Py_DECREF(owner);
                         PyGILState_Release(g);
                       })
                       .target_device(device)
                       .options(at::TensorOptions().dtype(at::kByte).device(device))
                       .make_tensor();
    return THPVariable_Wrap(std::move(t));
  } catch (const std::exception &e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

// part(tensor, offset, length): the bytes [offset, offset + length) of a uint8 tensor made by wrap
static PyObject *part(PyObject *, PyObject *const *args, Py_ssize_t n) {
  if (n != 3 || !THPVariable_Check(args[0])) {
    PyErr_SetString(PyExc_TypeError, "part(tensor, offset, length)");
    return nullptr;
  }
  const long long off = PyLong_AsLongLong(args[1]), len = PyLong_AsLongLong(args[2]);
  if (PyErr_Occurred()) return nullptr;
  const at::Tensor &t = THPVariable_Unpack(args[0]);
  if (off < 0 || len < 0 || t.dim() != 1 || off + len > t.numel()) {
    PyErr_SetString(PyExc_IndexError, "part: outside the tensor");
    return nullptr;
  }
  at::Tensor r = at::detail::make_tensor<c10::TensorImpl>(c10::TensorImpl::VIEW, c10::Storage(t.storage()),
                                                          t.key_set(), t.dtype());
  c10::TensorImpl *impl = r.unsafeGetTensorImpl();
  impl->set_storage_offset(t.storage_offset() + off);
  impl->set_sizes_contiguous(at::IntArrayRef{(int64_t)len});
  return THPVariable_Wrap(std::move(r));
}

static PyMethodDef methods[] = {
    {"wrap", (PyCFunction)(void (*)(void))wrap, METH_FASTCALL, "uint8 CUDA tensor over an address"},
    {"part", (PyCFunction)(void (*)(void))part, METH_FASTCALL, "part of a uint8 tensor"},
    {nullptr, nullptr, 0, nullptr}};
static PyModuleDef module = {PyModuleDef_HEAD_INIT, "_views", nullptr, -1, methods};
PyMODINIT_FUNC PyInit__views() { return PyModule_Create(&module); }
