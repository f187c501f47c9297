// Host arrays of the entry points as packed bytes, for the Python binding: device pointers per layer and donor maps.
//
// A call passes up to twelve such arrays.  Packed in Python one of four tensors takes 0.8 us, most of it in the method
// call per tensor, and the smallest calls are bound by the host: here it takes 0.1 us.  (The smallest training step, four
// calls with 32 arrays of four layers: see kvp.py.)
#define PY_SSIZE_T_CLEAN
#include <torch/csrc/autograd/python_variable.h>

namespace {

// [tensor or None, ...] -> their data pointers (0 for None) as 64-bit integers
PyObject* pointers(PyObject*, PyObject* seq) {
  PyObject* fast = PySequence_Fast(seq, "expected a sequence of tensors");
  if (fast == nullptr) return nullptr;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(fast);
  PyObject* out = PyBytes_FromStringAndSize(nullptr, n * Py_ssize_t(sizeof(uint64_t)));
  uint64_t* dst = out == nullptr ? nullptr : reinterpret_cast<uint64_t*>(PyBytes_AS_STRING(out));
  bool ok = out != nullptr;
  for (Py_ssize_t i = 0; i < n && ok; ++i) {
    PyObject* o = PySequence_Fast_GET_ITEM(fast, i);
    if (o == Py_None) {
      dst[i] = 0;
    } else if (THPVariable_CheckExact(o)) {
      try {
        dst[i] = reinterpret_cast<uint64_t>(THPVariable_Unpack(o).data_ptr());
      } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        ok = false;
      }
    } else {   // subclasses and whatever else has the method
      PyObject* p = PyObject_CallMethod(o, "data_ptr", nullptr);
      dst[i] = p == nullptr ? 0 : PyLong_AsUnsignedLongLong(p);
      Py_XDECREF(p);
      ok = PyErr_Occurred() == nullptr;
    }
  }
  Py_DECREF(fast);
  if (!ok) Py_CLEAR(out);
  return out;
}

// [int, ...] -> 32-bit integers
PyObject* donors(PyObject*, PyObject* seq) {
  PyObject* fast = PySequence_Fast(seq, "expected a sequence of integers");
  if (fast == nullptr) return nullptr;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(fast);
  PyObject* out = PyBytes_FromStringAndSize(nullptr, n * Py_ssize_t(sizeof(int32_t)));
  int32_t* dst = out == nullptr ? nullptr : reinterpret_cast<int32_t*>(PyBytes_AS_STRING(out));
  bool ok = out != nullptr;
  for (Py_ssize_t i = 0; i < n && ok; ++i) {
    PyObject* o = PySequence_Fast_GET_ITEM(fast, i);
    PyObject* v = PyLong_CheckExact(o) ? Py_NewRef(o) : PyNumber_Long(o);
    const long long x = v == nullptr ? 0 : PyLong_AsLongLong(v);
    Py_XDECREF(v);
    ok = PyErr_Occurred() == nullptr;
    if (ok && (x < INT32_MIN || x > INT32_MAX)) {
      PyErr_SetString(PyExc_OverflowError, "donor does not fit a 32-bit integer");
      ok = false;
    }
    dst[i] = int32_t(x);
  }
  Py_DECREF(fast);
  if (!ok) Py_CLEAR(out);
  return out;
}

PyMethodDef methods[] = {{"pointers", pointers, METH_O, nullptr}, {"donors", donors, METH_O, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pack", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__pack() { return PyModule_Create(&module); }
