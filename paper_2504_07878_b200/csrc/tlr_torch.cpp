// Router.route's call without options, as one native call: the checks of h, the arguments of tlr_route and the views that are
// handed out.  Marshalling only, like binding.py, which does the same with ctypes where this declines (anything but plain
// tensors, whatever is no number for a threshold) or was not built.
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

// t[:n].data for a one-dimensional contiguous tensor of at least n elements: made anew on every call (a batch size that was not
// asked for before costs what the others do), by the tensor's own copy with another length -- a slice from Python takes four times as long.
at::Tensor head_of(const at::Tensor& t, int64_t n) {
  auto impl = t.unsafeGetTensorImpl()->shallow_copy_and_detach(c10::VariableVersion(0), /*allow_tensor_metadata_change=*/true);
  impl->set_sizes_contiguous(n);
  impl->set_allow_tensor_metadata_change(false);
  return at::Tensor(std::move(impl));
}

bool has_head(const at::Tensor& t, int64_t n) { return t.dim() == 1 && t.is_contiguous() && t.size(0) >= n; }

// heads(n, t, ...): head_of every tensor, None if one has none.
PyObject* heads(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  if (nargs < 1) Py_RETURN_NONE;
  const long long n = PyLong_AsLongLong(args[0]);
  if (PyErr_Occurred()) return nullptr;
  for (Py_ssize_t i = 1; i < nargs; ++i)
    if (n < 0 || !THPVariable_CheckExact(args[i]) || !has_head(THPVariable_Unpack(args[i]), n)) Py_RETURN_NONE;
  PyObject* result = PyTuple_New(nargs - 1);
  if (result == nullptr) return nullptr;
  try {
    for (Py_ssize_t i = 1; i < nargs; ++i) {
      PyObject* o = THPVariable_Wrap(head_of(THPVariable_Unpack(args[i]), n));
      if (o == nullptr) {
        Py_DECREF(result);
        return nullptr;
      }
      PyTuple_SET_ITEM(result, i - 1, o);
    }
    return result;
  } catch (const std::exception& e) {
    Py_DECREF(result);
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

// route(ctx, d, h, tau, token, conf, entropy, route_mask, routed_idx, routed_count, stream): the six outputs, the first four as
// new views of n rows; the status if tlr_route fails; None if this call is not for here.
constexpr int kFirstOut = 4, kViews = 4, kOuts = 6, kArgs = kFirstOut + kOuts + 1;
PyObject* route(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  if (nargs != kArgs || g_route == nullptr || !THPVariable_CheckExact(args[2])) Py_RETURN_NONE;
  for (int i = 0; i < kOuts; ++i)
    if (!THPVariable_CheckExact(args[kFirstOut + i])) Py_RETURN_NONE;
  void* ctx = PyLong_AsVoidPtr(args[0]);
  const long long d = PyLong_AsLongLong(args[1]);
  const double tau = PyFloat_AsDouble(args[3]);
  void* stream = PyLong_AsVoidPtr(args[kArgs - 1]);
  if (PyErr_Occurred()) {       // (ctypes has its own idea of what a number is, and says so)
    PyErr_Clear();
    Py_RETURN_NONE;
  }
  try {
    const at::Tensor& h = THPVariable_Unpack(args[2]);
    if (!h.is_cuda() || h.scalar_type() != at::kBFloat16 || h.dim() != 2 || !h.is_contiguous() || h.size(1) != d)
      Py_RETURN_NONE;
    const int64_t n = h.size(0);
    void* out[kOuts];
    for (int i = 0; i < kOuts; ++i) {
      const at::Tensor& t = THPVariable_Unpack(args[kFirstOut + i]);
      if (i < kViews && !has_head(t, n)) Py_RETURN_NONE;
      out[i] = t.mutable_data_ptr();
    }
    const void* h_ptr = h.const_data_ptr();
    at::Tensor view[kViews];
    for (int i = 0; i < kViews; ++i) view[i] = head_of(THPVariable_Unpack(args[kFirstOut + i]), n);
    tlr_status status;
    Py_BEGIN_ALLOW_THREADS      // (a full launch queue waits for the GPU; nothing that may throw stands in here)
    status = g_route(static_cast<tlr_ctx*>(ctx), h_ptr, static_cast<int32_t>(n), static_cast<float>(tau),
                     static_cast<int32_t*>(out[0]), static_cast<float*>(out[1]), static_cast<float*>(out[2]),
                     static_cast<uint8_t*>(out[3]), static_cast<int32_t*>(out[4]), static_cast<int32_t*>(out[5]), stream);
    Py_END_ALLOW_THREADS
    if (status != TLR_OK) return PyLong_FromLong(status);
    PyObject* result = PyTuple_New(kOuts);
    if (result == nullptr) return nullptr;
    for (int i = 0; i < kOuts; ++i) {
      PyObject* o = i < kViews ? THPVariable_Wrap(std::move(view[i])) : Py_NewRef(args[kFirstOut + i]);
      if (o == nullptr) {
        Py_DECREF(result);
        return nullptr;
      }
      PyTuple_SET_ITEM(result, i, o);
    }
    return result;
  } catch (const std::exception& e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

PyMethodDef methods[] = {{"bind", bind, METH_O, "the address of tlr_route"},
                         {"route", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(route)), METH_FASTCALL,
                          "one routing step"},
                         {"heads", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(heads)), METH_FASTCALL,
                          "views of the first n elements"},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_tlr_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__tlr_torch() {
  PyObject* m = PyModule_Create(&module);
  if (m != nullptr && PyModule_AddStringConstant(m, "built_for", TLR_TORCH_VERSION) != 0) Py_CLEAR(m);
  return m;
}
