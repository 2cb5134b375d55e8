// kvE_decode_step for Python callers that issue it token by token: argument checks and the call without the interpreter in
// between.  (One robot's decode loop is bound by the host: a token of a small cache takes the GPU 7 us.  Checks in Python and the
// conversion of ten arguments by ctypes took 2.9 us of the 6.3 us that a call took, 1.0 here; 7 tokens call by call 95 -> 82 us.)
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

using DecodeStep = int (*)(void*, int, const void*, const void*, const void*, void*, float*, float, int, void*);

// address of a contiguous device tensor; rows > 0: of bf16 [rows, 128]
bool address(PyObject* o, int64_t rows, void** p) {
  if (!THPVariable_Check(o)) {
    PyErr_SetString(PyExc_TypeError, "a tensor is wanted");
    return false;
  }
  const at::Tensor& t = THPVariable_Unpack(o);
  if (!t.is_cuda() || !t.is_contiguous() ||
      (rows > 0 && (t.scalar_type() != at::kBFloat16 || t.dim() != 2 || t.size(0) != rows || t.size(1) != 128))) {
    PyErr_SetNone(PyExc_AssertionError);
    return false;
  }
  *p = t.data_ptr();
  return true;
}

// int(o): a float or any other number is taken too
long whole_number(PyObject* o) {
  if (PyLong_Check(o)) return PyLong_AsLong(o);
  PyObject* n = PyNumber_Long(o);
  if (!n) return -1;
  const long x = PyLong_AsLong(n);
  Py_DECREF(n);
  return x;
}

// decode_step(function address, handle, S, device, layer, k_new, v_new, q, out, lse or None, scale, n_reserve, stream or None) -> status
PyObject* decode_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 13) {
    PyErr_SetString(PyExc_TypeError, "13 arguments are wanted");
    return nullptr;
  }
  try {
    const auto fn = reinterpret_cast<DecodeStep>(PyLong_AsVoidPtr(a[0]));
    void* handle = a[1] == Py_None ? nullptr : PyLong_AsVoidPtr(a[1]);
    const long rows = PyLong_AsLong(a[2]), device = PyLong_AsLong(a[3]), layer = PyLong_AsLong(a[4]);
    const double scale = PyFloat_AsDouble(a[10]);
    const long n_reserve = whole_number(a[11]);
    void* stream = a[12] == Py_None ? nullptr : PyLong_AsVoidPtr(a[12]);
    if (PyErr_Occurred()) return nullptr;
    if (layer != (int)layer || n_reserve != (int)n_reserve) {
      PyErr_SetString(PyExc_OverflowError, "layer or n_reserve");
      return nullptr;
    }
    if (a[12] == Py_None) stream = c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)device).stream();
    void *k, *v, *q, *out, *lse = nullptr;
    if (!address(a[5], rows, &k) || !address(a[6], rows, &v) || !address(a[7], rows, &q) || !address(a[8], 0, &out)) return nullptr;
    if (a[9] != Py_None && !address(a[9], 0, &lse)) return nullptr;
    int rc;
    Py_BEGIN_ALLOW_THREADS      // a launch may wait for room in the queue
    rc = fn(handle, (int)layer, k, v, q, out, static_cast<float*>(lse), (float)scale, (int)n_reserve, stream);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

PyMethodDef methods[] = {{"decode_step", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(decode_step)), METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_kve_bind", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__kve_bind() { return PyModule_Create(&module); }
