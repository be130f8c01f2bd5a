// Calls of the C ABI from Python: argument marshalling and the call itself in native code.  A repair call of a small context is bound
// by the host: through ctypes, with a Python-level data_ptr() per tensor and an array object per list, the attention call took it
// 11.2 us (7.4 of them in the library, for two launches), the cache update 6.3 (3.9), the schedule 6.0 and the selection 5.2 (3.5);
// here 7.6, 4.1, 3.9 and 3.1.  One layer of 1 K tokens from selection to cache update 52.9 -> 48.2 us, of 16 K 109.5 -> 107.4.
//
//   marshal(codes, ...)          the arguments of an entry point: 'p' an object with data_ptr() (or None) -> its address, 'h' host
//                                integers (or None) -> bytes that hold them as int32, 's' a ctypes structure -> its address,
//                                '.' anything, as it is.
//   bind(name, address, other)   the entry point at `address` as a callable over integers, floats, bytes and None.  A call with
//                                anything else among its arguments (a ctypes reference, a wrong count) is `other`'s.
// The interpreter's lock is released during the call, as ctypes does it.  Python 3.10 or newer.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <structmember.h>                                  // T_PYSSIZET, READONLY: the names that Python 3.10 and 3.11 have, too
#include <cstddef>
#include <cstdint>
#include <cstring>
#include <tuple>
#include <type_traits>
#include <utility>
#include "relaxkv.h"

namespace {

PyObject* g_data_ptr;                                      // the interned name "data_ptr"

// ---- marshal ------------------------------------------------------------------------------------------------------------------

PyObject* host_ints(PyObject* xs) {
  if (PyObject_Size(xs) < 0) return nullptr;               // what has no length is refused, as ever
  PyObject* seq = PySequence_Fast(xs, "host integers expected");
  if (!seq) return nullptr;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
  PyObject* out = PyBytes_FromStringAndSize(nullptr, n * 4);
  for (Py_ssize_t i = 0; out && i < n; ++i) {
    // (the size is looked at again: a list may change while an element's own conversion runs)
    PyObject* item = i < PySequence_Fast_GET_SIZE(seq) ? PySequence_Fast_GET_ITEM(seq, i) : nullptr;
    if (!item) PyErr_SetString(PyExc_RuntimeError, "host integers changed size");
    Py_XINCREF(item);
    PyObject* num = item ? (PyLong_CheckExact(item) ? Py_NewRef(item) : PyNumber_Long(item)) : nullptr;
    Py_XDECREF(item);
    if (!num) { Py_CLEAR(out); break; }
    const int32_t v = (int32_t)PyLong_AsUnsignedLongMask(num);
    Py_DECREF(num);
    memcpy(PyBytes_AS_STRING(out) + 4 * i, &v, 4);
  }
  Py_DECREF(seq);
  return out;
}

PyObject* struct_address(PyObject* s) {
  Py_buffer b;
  if (PyObject_GetBuffer(s, &b, PyBUF_SIMPLE) < 0) return nullptr;
  PyObject* out = PyLong_FromVoidPtr(b.buf);
  PyBuffer_Release(&b);                                    // a ctypes structure keeps its memory as long as it lives
  return out;
}

PyObject* marshal(PyObject*, PyObject* const* args, Py_ssize_t n) {
  Py_ssize_t n_codes = 0;
  const char* codes = n > 0 ? PyUnicode_AsUTF8AndSize(args[0], &n_codes) : nullptr;
  if (!codes) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "marshal(codes, ...)");
    return nullptr;
  }
  if (n_codes != n - 1) return PyErr_Format(PyExc_TypeError, "marshal: %zd codes for %zd arguments", n_codes, n - 1);
  PyObject* out = PyTuple_New(n_codes);
  for (Py_ssize_t i = 0; out && i < n_codes; ++i) {
    PyObject* a = args[i + 1];
    PyObject* v = nullptr;
    if (codes[i] == '.' || (a == Py_None && codes[i] != 's')) v = Py_NewRef(a);
    else if (codes[i] == 'p') v = PyObject_CallMethodNoArgs(a, g_data_ptr);
    else if (codes[i] == 'h') v = host_ints(a);
    else if (codes[i] == 's') v = struct_address(a);
    else PyErr_Format(PyExc_TypeError, "marshal: code '%c'", codes[i]);
    if (!v) { Py_CLEAR(out); break; }
    PyTuple_SET_ITEM(out, i, v);
  }
  return out;
}

// ---- bind ---------------------------------------------------------------------------------------------------------------------

// One argument as the C type; false: not a form that is taken here.
template <class T>
bool convert(PyObject* a, T* out) {
  if constexpr (std::is_pointer_v<T>) {
    if (a == Py_None) *out = nullptr;
    else if (PyLong_Check(a)) *out = reinterpret_cast<T>((uintptr_t)PyLong_AsUnsignedLongLongMask(a));
    else if (PyBytes_Check(a)) *out = reinterpret_cast<T>(PyBytes_AS_STRING(a));
    else return false;
  } else if constexpr (std::is_floating_point_v<T>) {
    if (PyFloat_Check(a)) *out = (T)PyFloat_AS_DOUBLE(a);
    else return false;
  } else {
    if (!PyLong_Check(a)) return false;
    *out = (T)PyLong_AsUnsignedLongLongMask(a);
  }
  return true;
}

struct Entry {
  PyObject_HEAD
  vectorcallfunc vectorcall;
  void* fn;
  PyObject* other;
};

template <class F>
struct Call;
template <class... A>
struct Call<relaxkv_status (*)(A...)> {
  static PyObject* vectorcall(PyObject* self, PyObject* const* args, size_t nargsf, PyObject* kw) {
    return run(reinterpret_cast<Entry*>(self), args, nargsf, kw, std::index_sequence_for<A...>{});
  }
  template <size_t... I>
  static PyObject* run(Entry* e, PyObject* const* args, size_t nargsf, PyObject* kw, std::index_sequence<I...>) {
    std::tuple<A...> v;
    if (kw || PyVectorcall_NARGS(nargsf) != (Py_ssize_t)sizeof...(A) || !(convert(args[I], &std::get<I>(v)) && ...))
      return PyObject_Vectorcall(e->other, args, nargsf, kw);
    relaxkv_status rc;
    Py_BEGIN_ALLOW_THREADS
    rc = reinterpret_cast<relaxkv_status (*)(A...)>(e->fn)(std::get<I>(v)...);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong((long)rc);
  }
};

struct Known { const char* name; vectorcallfunc call; };
#define KNOWN(f) {#f, Call<decltype(&f)>::vectorcall}
const Known kKnown[] = {
    KNOWN(relaxkv_select_topk), KNOWN(relaxkv_build_active_sets), KNOWN(relaxkv_build_active_sets_static),
    KNOWN(relaxkv_sparse_ctx_attention), KNOWN(relaxkv_scatter_kv), KNOWN(relaxkv_gather_kv), KNOWN(relaxkv_list_attention),
    KNOWN(relaxkv_cache_attention), KNOWN(relaxkv_scatter_kv_lists), KNOWN(relaxkv_query_prefill_attention), KNOWN(relaxkv_rmsnorm),
    KNOWN(relaxkv_linear), KNOWN(relaxkv_linear_qkv), KNOWN(relaxkv_linear_swiglu), KNOWN(relaxkv_qk_norm_rope),
    KNOWN(relaxkv_qk_norm_rope_append), KNOWN(relaxkv_swiglu), KNOWN(relaxkv_target_positions), KNOWN(relaxkv_carry_rows),
};

void entry_dealloc(PyObject* self) {
  PyTypeObject* type = Py_TYPE(self);
  Py_XDECREF(reinterpret_cast<Entry*>(self)->other);
  type->tp_free(self);
  Py_DECREF(type);
}

PyMemberDef entry_members[] = {
    {"__vectorcalloffset__", T_PYSSIZET, offsetof(Entry, vectorcall), READONLY, nullptr}, {nullptr, 0, 0, 0, nullptr}};
PyType_Slot entry_slots[] = {{Py_tp_dealloc, (void*)entry_dealloc}, {Py_tp_call, (void*)PyVectorcall_Call},
                             {Py_tp_members, entry_members}, {0, nullptr}};
PyType_Spec entry_spec = {"paper_2609_33503_b200._calls.Entry", sizeof(Entry), 0,
                          Py_TPFLAGS_DEFAULT | Py_TPFLAGS_HAVE_VECTORCALL | Py_TPFLAGS_DISALLOW_INSTANTIATION, entry_slots};
PyTypeObject* g_entry_type;

PyObject* bind(PyObject*, PyObject* args) {
  const char* name;
  unsigned long long address;
  PyObject* other;
  if (!PyArg_ParseTuple(args, "sKO", &name, &address, &other)) return nullptr;
  for (const Known& k : kKnown) {
    if (strcmp(k.name, name)) continue;
    Entry* e = PyObject_New(Entry, g_entry_type);
    if (!e) return nullptr;
    e->vectorcall = k.call;
    e->fn = reinterpret_cast<void*>((uintptr_t)address);
    e->other = Py_NewRef(other);
    return reinterpret_cast<PyObject*>(e);
  }
  return Py_NewRef(other);
}

PyMethodDef methods[] = {{"marshal", (PyCFunction)(void (*)())marshal, METH_FASTCALL, nullptr}, {"bind", bind, METH_VARARGS, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() {
  g_data_ptr = PyUnicode_InternFromString("data_ptr");
  g_entry_type = reinterpret_cast<PyTypeObject*>(PyType_FromSpec(&entry_spec));
  return g_data_ptr && g_entry_type ? PyModule_Create(&module) : nullptr;
}
