// Tensors over memory the library owns, made without the interpreter's indexing machinery: a
// result has up to nineteen columns, and taking a slice of a tensor from Python costs 1.4 us (here
// 0.2), wrapping an address through __cuda_array_interface__ eight.
#include <Python.h>

#include <ATen/ops/from_blob.h>
#include <c10/core/InferenceMode.h>
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
    const c10::InferenceMode plain(false);  // usable outside the caller's inference mode as well
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

// part((first address, address behind, tensor made by wrap), address, nbytes): those bytes of the
// tensor as one of its own, None if they are not its
static PyObject *part(PyObject *, PyObject *const *args, Py_ssize_t n) {
  if (n != 3 || !PyTuple_Check(args[0]) || PyTuple_GET_SIZE(args[0]) != 3) {
    PyErr_SetString(PyExc_TypeError, "part((first, behind, tensor), address, nbytes)");
    return nullptr;
  }
  const unsigned long long lo = PyLong_AsUnsignedLongLong(PyTuple_GET_ITEM(args[0], 0)),
                           hi = PyLong_AsUnsignedLongLong(PyTuple_GET_ITEM(args[0], 1)),
                           at = PyLong_AsUnsignedLongLong(args[1]), len = PyLong_AsUnsignedLongLong(args[2]);
  if (PyErr_Occurred()) return nullptr;
  PyObject *base = PyTuple_GET_ITEM(args[0], 2);
  if (at < lo || at > hi || len > hi - at || !THPVariable_Check(base)) Py_RETURN_NONE;
  try {
    const at::Tensor &t = THPVariable_Unpack(base);
    if (t.dim() != 1 || (unsigned long long)t.numel() != hi - lo) {
      PyErr_SetString(PyExc_ValueError, "part: not a tensor of these bytes");
      return nullptr;
    }
    at::Tensor r = at::detail::make_tensor<c10::TensorImpl>(c10::TensorImpl::VIEW, c10::Storage(t.storage()),
                                                            t.key_set(), t.dtype());
    c10::TensorImpl *impl = r.unsafeGetTensorImpl();
    impl->set_storage_offset(t.storage_offset() + (int64_t)(at - lo));
    impl->set_sizes_contiguous(at::IntArrayRef{(int64_t)len});
    return THPVariable_Wrap(std::move(r));
  } catch (const std::exception &e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

static PyMethodDef methods[] = {
    {"wrap", (PyCFunction)(void (*)(void))wrap, METH_FASTCALL, "uint8 CUDA tensor over an address"},
    {"part", (PyCFunction)(void (*)(void))part, METH_FASTCALL, "part of a uint8 tensor"},
    {nullptr, nullptr, 0, nullptr}};
static PyModuleDef module = {PyModuleDef_HEAD_INIT, "_views", nullptr, -1, methods};
PyMODINIT_FUNC PyInit__views() { return PyModule_Create(&module); }
