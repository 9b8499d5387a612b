// The call a program makes once per layer and pass, WinogradConv.forward, on torch tensors:
// allocates the output and calls wino_conv_forward on torch's current stream.  Argument
// marshalling only, as in wino_python.c; being compiled against torch it reads tensor addresses
// and allocates through the caching allocator without going through Python and the dispatcher,
// which took 2.3 of the 5.5 us of a small layer's pass.
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include "wino.h"

namespace {

bool tensor_or_none(PyObject* o) { return o == Py_None || THPVariable_Check(o); }
void* address(PyObject* o) { return o == Py_None ? nullptr : THPVariable_Unpack(o).mutable_data_ptr(); }

// (plan, x, U_q, bias, y or None, workspace, like) -> y, the (negative) return code, or None where
// an argument is not a tensor.  like: a tensor of the output's shape, type and device.
PyObject* forward(PyObject*, PyObject* const* a, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  if (n != 7) {
    PyErr_Format(PyExc_TypeError, "forward takes 7 arguments (%zd given)", n);
    return nullptr;
  }
  for (int i = 1; i < 6; ++i)
    if (!tensor_or_none(a[i])) Py_RETURN_NONE;
  if (!THPVariable_Check(a[6])) Py_RETURN_NONE;
  void* plan = PyLong_AsVoidPtr(a[0]);
  if (plan == nullptr && PyErr_Occurred()) return nullptr;
  PyObject* result;
  void* y;
  if (a[4] == Py_None) {
    const at::Tensor& like = THPVariable_Unpack(a[6]);
    at::Tensor out = at::detail::empty_cuda(like.sizes(), like.scalar_type(), like.device(), std::nullopt);
    y = out.mutable_data_ptr();
    result = THPVariable_Wrap(std::move(out));
    if (result == nullptr) return nullptr;
  } else {
    y = address(a[4]);
    result = Py_NewRef(a[4]);
  }
  const void* x = address(a[1]);
  const void* u = address(a[2]);
  const void* bias = address(a[3]);
  void* ws = address(a[5]);
  cudaStream_t st = c10::cuda::getCurrentCUDAStream().stream();
  int rc;
  Py_BEGIN_ALLOW_THREADS   // a launch may wait for room in the queue
  rc = wino_conv_forward(static_cast<wino_plan_t*>(plan), static_cast<const int8_t*>(x), static_cast<const int8_t*>(u),
                         static_cast<const float*>(bias), y, ws, st);
  Py_END_ALLOW_THREADS
  if (rc == WINO_OK) return result;
  Py_DECREF(result);
  return PyLong_FromLong(rc);
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"forward", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(forward)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__native_torch(void) { return PyModule_Create(&module); }
