// The C ABI's calls of a training iteration as Python functions: the arguments of include/ard.h in their order, device
// memory as torch tensors (data_ptr() is asked for here), integers or None, handles as ctypes.c_void_p.  Returns the ard_status.
//
// An iteration of a small layer is bound by the host: a call through ctypes spent 2.9 us on its arguments where the native
// call behind it takes 4.
#include <Python.h>

#include <stdint.h>

#include <tuple>
#include <utility>

#include "ard.h"

namespace {

PyObject *g_void_p, *g_data_ptr;  // ctypes.c_void_p; the method's name

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
template <typename T>
bool convert(PyObject* o, T*& v) {
  if (o == Py_None) {
    v = nullptr;
    return true;
  }
  if ((PyObject*)Py_TYPE(o) == g_void_p) {  // its memory holds the pointer
    Py_buffer b;
    if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
    v = *(T**)b.buf;
    PyBuffer_Release(&b);
    return true;
  }
  uint64_t x;
  if (PyLong_Check(o)) {
    if (!convert(o, x)) return false;
  } else {
    PyObject* p = PyObject_CallMethodNoArgs(o, g_data_ptr);
    if (p == nullptr) return false;
    const bool ok = convert(p, x);
    Py_DECREF(p);
    if (!ok) return false;
  }
  v = (T*)(uintptr_t)x;
  return true;
}

template <typename... A, size_t... I>
PyObject* call(ard_status (*f)(A...), PyObject* const* args, std::index_sequence<I...>) {
  std::tuple<std::remove_const_t<A>...> v;
  if (!(convert(args[I], std::get<I>(v)) && ...)) return nullptr;
  ard_status st;
  Py_BEGIN_ALLOW_THREADS
  st = f(std::get<I>(v)...);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong((long)st);
}
template <typename... A>
PyObject* call(ard_status (*f)(A...), PyObject* const* args, Py_ssize_t n) {
  if (n != (Py_ssize_t)sizeof...(A)) {
    PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", (Py_ssize_t)sizeof...(A), n);
    return nullptr;
  }
  return call(f, args, std::index_sequence_for<A...>{});
}
template <auto F>
PyObject* entry(PyObject*, PyObject* const* args, Py_ssize_t n) {
  return call(F, args, n);
}

#define CALL(name) {#name, (PyCFunction)(void (*)(void))entry<&name>, METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
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
