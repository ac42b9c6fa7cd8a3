// Router.route's call without options, as one native call: the checks of h, the arguments of tlr_route and the views that are
// handed out.  Marshalling only, like binding.py, which does the same with ctypes where this declines (anything but a plain
// tensor; whatever is no number for a threshold; a batch size whose views are not made yet) or was not built.
// A step of a small batch takes the GPU less time than it took the interpreter to ask for it: n = 1, d = 256, V = 20000
// 8.9 us per call through ctypes, 5.6 of them tlr_route and its two launches.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <torch/csrc/autograd/python_variable.h>

#include "tlr.h"

namespace {

using RouteFn = decltype(&tlr_route);
RouteFn g_route = nullptr;

PyObject* bind(PyObject*, PyObject* address) {
  g_route = reinterpret_cast<RouteFn>(PyLong_AsVoidPtr(address));
  if (PyErr_Occurred()) return nullptr;
  Py_RETURN_NONE;
}

template <class T>
T* data_of(PyObject* tensor) {
  return static_cast<T*>(THPVariable_Unpack(tensor).mutable_data_ptr());
}

// route(ctx, d, h, tau, views, routed_idx, routed_count, stream): views maps a batch size to (token, conf, entropy, route_mask).
// The six outputs as new views; the status if tlr_route fails; None if this call is not for here.
PyObject* route(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  if (nargs != 8 || g_route == nullptr) Py_RETURN_NONE;
  PyObject *h_obj = args[2], *idx_obj = args[5], *count_obj = args[6];
  if (!THPVariable_CheckExact(h_obj) || !THPVariable_CheckExact(idx_obj) || !THPVariable_CheckExact(count_obj) ||
      !PyDict_CheckExact(args[4]))
    Py_RETURN_NONE;
  try {
    void* ctx = PyLong_AsVoidPtr(args[0]);
    const long long d = PyLong_AsLongLong(args[1]);
    const double tau = PyFloat_AsDouble(args[3]);
    void* stream = PyLong_AsVoidPtr(args[7]);
    if (PyErr_Occurred()) {       // (ctypes has its own idea of what a number is, and says so)
      PyErr_Clear();
      Py_RETURN_NONE;
    }
    const at::Tensor& h = THPVariable_Unpack(h_obj);
    if (!h.is_cuda() || h.scalar_type() != at::kBFloat16 || h.dim() != 2 || !h.is_contiguous() || h.size(1) != d)
      Py_RETURN_NONE;
    const int64_t n = h.size(0);
    PyObject* key = PyLong_FromLongLong(n);
    if (key == nullptr) return nullptr;
    PyObject* kept = PyDict_GetItemWithError(args[4], key);      // (borrowed)
    Py_DECREF(key);
    if (kept == nullptr) {
      if (PyErr_Occurred()) return nullptr;
      Py_RETURN_NONE;
    }
    if (!PyTuple_CheckExact(kept) || PyTuple_GET_SIZE(kept) != 4) Py_RETURN_NONE;
    at::Tensor view[4];
    for (int i = 0; i < 4; ++i) {
      if (!THPVariable_CheckExact(PyTuple_GET_ITEM(kept, i))) Py_RETURN_NONE;
      view[i] = THPVariable_Unpack(PyTuple_GET_ITEM(kept, i)).variable_data();
    }
    void* rows[4];
    for (int i = 0; i < 4; ++i) rows[i] = view[i].mutable_data_ptr();
    const void* h_ptr = h.const_data_ptr();
    int32_t* idx = data_of<int32_t>(idx_obj);
    int32_t* count = data_of<int32_t>(count_obj);
    tlr_status status;
    Py_BEGIN_ALLOW_THREADS      // (a full launch queue waits for the GPU; nothing that may throw stands in here)
    status = g_route(static_cast<tlr_ctx*>(ctx), h_ptr, static_cast<int32_t>(n), static_cast<float>(tau),
                     static_cast<int32_t*>(rows[0]), static_cast<float*>(rows[1]), static_cast<float*>(rows[2]),
                     static_cast<uint8_t*>(rows[3]), idx, count, stream);
    Py_END_ALLOW_THREADS
    if (status != TLR_OK) return PyLong_FromLong(status);
    PyObject* out = PyTuple_New(6);
    if (out == nullptr) return nullptr;
    for (int i = 0; i < 4; ++i) {
      PyObject* o = THPVariable_Wrap(view[i]);
      if (o == nullptr) {
        Py_DECREF(out);
        return nullptr;
      }
      PyTuple_SET_ITEM(out, i, o);
    }
    Py_INCREF(idx_obj);
    Py_INCREF(count_obj);
    PyTuple_SET_ITEM(out, 4, idx_obj);
    PyTuple_SET_ITEM(out, 5, count_obj);
    return out;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

PyMethodDef methods[] = {{"bind", bind, METH_O, "the address of tlr_route"},
                         {"route", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(route)), METH_FASTCALL,
                          "one routing step"},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_tlr_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__tlr_torch() {
  PyObject* m = PyModule_Create(&module);
  if (m != nullptr && PyModule_AddStringConstant(m, "built_for", TLR_TORCH_VERSION) != 0) Py_CLEAR(m);
  return m;
}
