// The C ABI's calls of a training iteration as Python functions: the arguments of include/ard.h in their order, device
// memory as torch tensors (data_ptr() is asked for here), integers or None, handles as ctypes.c_void_p.  Returns the ard_status.
// Arguments of any other kind go to the function given to fall_back(), which makes the call through ctypes: that takes, or refuses
// in its own words, whatever it always did.
//
// An iteration of a small layer is bound by the host: a call through ctypes spent 2.9 us on its arguments where the native
// call behind it takes 4.
#include <Python.h>

#include <stdint.h>

#include <tuple>
#include <type_traits>
#include <utility>

#include "ard.h"

namespace {

PyObject *g_void_p, *g_data_ptr;  // ctypes.c_void_p; the method's name
PyObject* g_fall_back;            // (name, arguments...)

// Each convert() returns false for what it does not take, an error set or not.

bool convert(PyObject* o, int& v) {
  const unsigned long x = PyLong_AsUnsignedLongMask(o);  // what does not fit is cut off, as ctypes does
  if (x == (unsigned long)-1 && PyErr_Occurred()) return false;
  v = (int)(uint32_t)x;
  return true;
}
bool convert(PyObject* o, uint32_t& v) {
  int x;
  if (!convert(o, x)) return false;
  v = (uint32_t)x;
  return true;
}
bool convert(PyObject* o, uint64_t& v) {
  v = PyLong_AsUnsignedLongLongMask(o);
  return !(v == (uint64_t)-1 && PyErr_Occurred());
}
bool convert(PyObject* o, double& v) {
  v = PyFloat_AsDouble(o);
  return !(v == -1.0 && PyErr_Occurred());
}
bool convert(PyObject* o, float& v) {
  double x;
  if (!convert(o, x)) return false;
  v = (float)x;
  return true;
}
template <typename E, std::enable_if_t<std::is_enum<E>::value, int> = 0>
bool convert(PyObject* o, E& v) {
  int x;
  if (!convert(o, x)) return false;
  v = (E)x;
  return true;
}
// Handles and streams
template <typename T>
bool convert_handle(PyObject* o, T*& v) {
  if (o == Py_None) {
    v = nullptr;
    return true;
  }
  uint64_t x;
  if ((PyObject*)Py_TYPE(o) == g_void_p) {  // its memory holds the pointer
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
    v = *(T**)b.buf;
    PyBuffer_Release(&b);
    return true;
  }
  if (!PyLong_Check(o) || !convert(o, x)) return false;
  v = (T*)(uintptr_t)x;
  return true;
}
bool convert(PyObject* o, ard_ctx*& v) { return convert_handle(o, v); }
bool convert(PyObject* o, const ard_pattern*& v) { return convert_handle(o, v); }
bool convert(PyObject* o, ard_pattern*& v) { return convert_handle(o, v); }
bool convert(PyObject* o, const ard_rows*& v) { return convert_handle(o, v); }
bool convert(PyObject* o, ard_rows*& v) { return convert_handle(o, v); }
bool convert(PyObject* o, const ard_blocks*& v) { return convert_handle(o, v); }
bool convert(PyObject* o, ard_blocks*& v) { return convert_handle(o, v); }
// Device memory
template <typename T>
bool convert(PyObject* o, T*& v) {
  if (o == Py_None) {
    v = nullptr;
    return true;
  }
  uint64_t x;
  if (PyLong_Check(o)) {
    if (!convert(o, x)) return false;
  } else {
    PyObject* p = PyObject_CallMethodNoArgs(o, g_data_ptr);
    if (p == nullptr) return false;
    const bool ok = PyLong_Check(p) && convert(p, x);
    Py_DECREF(p);
    if (!ok) return false;
  }
  v = (T*)(uintptr_t)x;
  return true;
}
// Argument i of n: a pointer in the last place is the stream.
template <typename T>
bool convert_argument(PyObject* o, T& v, size_t i, size_t n) {
  if constexpr (std::is_same<T, void*>::value) {
    if (i + 1 == n) return convert_handle(o, v);
  }
  return convert(o, v);
}

template <typename... A, size_t... I>
PyObject* call(ard_status (*f)(A...), const char* name, PyObject* const* args, std::index_sequence<I...>) {
  std::tuple<std::remove_const_t<A>...> v;
  if (!(convert_argument(args[I], std::get<I>(v), I, sizeof...(A)) && ...)) {
    if (g_fall_back == nullptr) {
      if (!PyErr_Occurred()) PyErr_Format(PyExc_TypeError, "%s: argument of a type that is not taken", name);
      return nullptr;
    }
    PyErr_Clear();
    PyObject* n = PyUnicode_FromString(name);
    if (n == nullptr) return nullptr;
    PyObject* all[] = {n, args[I]...};
    PyObject* r = PyObject_Vectorcall(g_fall_back, all, 1 + sizeof...(A), nullptr);
    Py_DECREF(n);
    return r;
  }
  ard_status st;
  Py_BEGIN_ALLOW_THREADS
  st = f(std::get<I>(v)...);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong((long)st);
}
template <typename... A>
PyObject* call(ard_status (*f)(A...), const char* name, PyObject* const* args, Py_ssize_t n) {
  if (n != (Py_ssize_t)sizeof...(A)) {
    PyErr_Format(PyExc_TypeError, "%s: %zd arguments expected, %zd given", name, (Py_ssize_t)sizeof...(A), n);
    return nullptr;
  }
  return call(f, name, args, std::index_sequence_for<A...>{});
}
PyObject* fall_back(PyObject*, PyObject* f) {
  Py_INCREF(f);
  Py_XSETREF(g_fall_back, f);
  Py_RETURN_NONE;
}

#define CALL(name)                                                                                            \
  {#name, (PyCFunction)(void (*)(void))+[](PyObject*, PyObject* const* a, Py_ssize_t n) { return call(&name, #name, a, n); }, \
   METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    {"fall_back", fall_back, METH_O, nullptr},
    CALL(ard_sample_pattern), CALL(ard_sample_pattern_counter), CALL(ard_pattern_set), CALL(ard_fwd), CALL(ard_bwd_data),
    CALL(ard_bwd_weight), CALL(ard_bwd_data_static_scratch), CALL(ard_layer_fwd), CALL(ard_layer_bwd_data),
    CALL(ard_layer_bwd_weight), CALL(ard_layer_products), CALL(ard_compact_weight_cols), CALL(ard_expand_weight_grad_cols),
    CALL(ard_bias_grad), CALL(ard_compact_cols), CALL(ard_expand_cols), CALL(ard_lstm_forward), CALL(ard_lstm_backward),
    CALL(ard_lstm_backward_dh), CALL(ard_lstm_forward_from_gates), CALL(ard_lstm_backward_recurrent), CALL(ard_lstm_gates),
    CALL(ard_lstm_gates_bwd), CALL(ard_lstm_gate_gemm), CALL(ard_lstm_gate_gemm_bwd), CALL(ard_sensitivity_predict),
    CALL(ard_rows_sample), CALL(ard_rows_products), CALL(ard_rows_gather), CALL(ard_rows_fwd), CALL(ard_rows_bwd_data),
    CALL(ard_rows_bwd_weight), CALL(ard_rows_fwd_compact), CALL(ard_rows_bwd_data_compact), CALL(ard_rows_bwd_weight_compact),
    CALL(ard_blocks_predict), CALL(ard_blocks_sample), CALL(ard_blocks_fwd), CALL(ard_blocks_bwd_weight),
    CALL(ard_blocks_bwd_input), CALL(ard_blocks_products), {nullptr, nullptr, 0, nullptr}};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls(void) {
  PyObject* ctypes = PyImport_ImportModule("ctypes");
  if (ctypes == nullptr) return nullptr;
  g_void_p = PyObject_GetAttrString(ctypes, "c_void_p");
  Py_DECREF(ctypes);
  g_data_ptr = PyUnicode_InternFromString("data_ptr");
  if (g_void_p == nullptr || g_data_ptr == nullptr) return nullptr;
  return PyModule_Create(&g_module);
}
