// CPython side of the binding: the C entry points as functions that take tensors, numbers and lists as specvlm.py has
// them.  ctypes spends 1.0 us on a call of eleven arguments, a microsecond on a list of integers per sequence
// and 0.1 us on each tensor's address, of 5 to 8 us that a short call takes on the host.
//
// Every function takes the C arguments in order without the stream, which is the current one of the current device:
//   KvStruct    its address (int)       device pointer   a tensor (its data_ptr()) or None; a number is refused
//   host array  any sequence of integers; integers are taken modulo 2^32, as ctypes takes them
// and returns the status.  The interpreter lock is released during the call.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstdint>
#include <tuple>
#include <utility>
#include <vector>

#include "../../include/specvlm.h"

namespace {

PyObject* g_get_device = nullptr;      // torch._C._cuda_getDevice
PyObject* g_get_raw_stream = nullptr;  // torch._C._cuda_getCurrentRawStream
PyObject* g_data_ptr = nullptr;        // "data_ptr"

struct AnyPtr {
  void* p;
  template <typename T> operator T*() const { return static_cast<T*>(p); }
};

// One class per kind of argument: set() converts, get() is what the C function takes.
struct Kv {
  static constexpr int kArgs = 1;
  const specvlm_kv_t* v = nullptr;
  bool set(PyObject* o) {
    v = static_cast<const specvlm_kv_t*>(PyLong_AsVoidPtr(o));
    return !PyErr_Occurred();
  }
  const specvlm_kv_t* get() const { return v; }
};
struct Ptr {
  static constexpr int kArgs = 1;
  void* v = nullptr;
  bool set(PyObject* o) {
    if (o == Py_None) return true;
    PyObject* const a = PyObject_CallMethodNoArgs(o, g_data_ptr);
    if (!a) return false;
    v = PyLong_AsVoidPtr(a);
    Py_DECREF(a);
    return !PyErr_Occurred();
  }
  AnyPtr get() const { return {v}; }
};
// An integer, or what stands for one (__index__: numpy's integers, tensors of one integer); a float is none.
bool to_int(PyObject* o, unsigned long long& v) {
  v = PyLong_AsUnsignedLongLongMask(o);
  return !PyErr_Occurred();
}
template <typename T>
struct Int {
  static constexpr int kArgs = 1;
  T v = 0;
  bool set(PyObject* o) {
    unsigned long long x;
    if (!to_int(o, x)) return false;
    v = static_cast<T>(x);
    return true;
  }
  T get() const { return v; }
};
struct Float {
  static constexpr int kArgs = 1;
  float v = 0.f;
  bool set(PyObject* o) {
    v = static_cast<float>(PyFloat_AsDouble(o));
    return !PyErr_Occurred();
  }
  float get() const { return v; }
};
struct Array {
  static constexpr int kArgs = 1;
  static constexpr int kSmall = 66;    // sequences of a call as a rule, and one more for running sums
  int32_t small[kSmall];
  std::vector<int32_t> big;
  int32_t* data = small;
  bool set(PyObject* o) {
    if (PyObject_Size(o) < 0) return false;
    PyObject* const seq = PySequence_Fast(o, "a sequence of integers is expected");
    if (!seq) return false;
    const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
    bool ok = true;
    if (n > kSmall) {
      try {
        big.resize(static_cast<size_t>(n));
      } catch (...) {
        PyErr_NoMemory();
        ok = false;
      }
      data = big.data();
    }
    for (Py_ssize_t i = 0; ok && i < n; ++i) {
      unsigned long long x = 0;
      // a list is read in place, and an element's conversion may run code (or let another thread run) that shortens it:
      // what is gone reads as 0, and the element is held while it is converted
      PyObject* const item = i < PySequence_Fast_GET_SIZE(seq) ? PySequence_Fast_GET_ITEM(seq, i) : nullptr;
      if (item && PyLong_CheckExact(item)) {
        ok = to_int(item, x);
      } else if (item) {
        Py_INCREF(item);
        PyObject* const whole = PyNumber_Long(item);
        Py_DECREF(item);
        ok = whole && to_int(whole, x);
        Py_XDECREF(whole);
      }
      if (ok) data[i] = static_cast<int32_t>(x);
    }
    Py_DECREF(seq);
    return ok;
  }
  int32_t* get() { return data; }
};
struct Stream {
  static constexpr int kArgs = 0;
  void* v = nullptr;
  bool set(PyObject*) {
    PyObject* const dev = g_get_device ? PyObject_CallNoArgs(g_get_device) : nullptr;
    if (!dev) {
      if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, "the binding has not been initialised");
      return false;
    }
    PyObject* const h = PyObject_CallOneArg(g_get_raw_stream, dev);
    Py_DECREF(dev);
    if (!h) return false;
    v = PyLong_AsVoidPtr(h);
    Py_DECREF(h);
    return !PyErr_Occurred();
  }
  AnyPtr get() const { return {v}; }
};

template <auto fn, typename... Kinds>
struct Entry {
  static constexpr Py_ssize_t kArgs = (Kinds::kArgs + ... + 0);
  template <size_t... I>
  static PyObject* run(PyObject* const* args, std::index_sequence<I...>) {
    std::tuple<Kinds...> a;
    Py_ssize_t at = 0;
    const bool ok = ([&] {
      using K = std::tuple_element_t<I, std::tuple<Kinds...>>;
      PyObject* const o = K::kArgs ? args[at] : nullptr;
      at += K::kArgs;
      return std::get<I>(a).set(o);
    }() && ...);
    if (!ok) return nullptr;
    int32_t rc;
    Py_BEGIN_ALLOW_THREADS
    rc = fn(std::get<I>(a).get()...);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
  }
  static PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t n) {
    if (n != kArgs) {
      PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", kArgs, n);
      return nullptr;
    }
    return run(args, std::index_sequence_for<Kinds...>{});
  }
};

PyObject* init(PyObject*, PyObject* const* args, Py_ssize_t n) {
  if (n != 2) {
    PyErr_SetString(PyExc_TypeError, "two functions expected");
    return nullptr;
  }
  for (int i = 0; i < 2; ++i) Py_INCREF(args[i]);
  Py_XSETREF(g_get_device, args[0]);
  Py_XSETREF(g_get_raw_stream, args[1]);
  Py_RETURN_NONE;
}

using I32 = Int<int32_t>;
using Size = Int<size_t>;
#define SPECVLM_ENTRY(name, ...) \
  {#name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&Entry<&specvlm_##name, __VA_ARGS__, Stream>::call)), METH_FASTCALL, nullptr}

PyMethodDef g_methods[] = {
    {"init", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(&init)), METH_FASTCALL, nullptr},
    SPECVLM_ENTRY(stage1_row_lse, Kv, Ptr, Array, Array, I32, I32, Float, Ptr, Ptr),
    SPECVLM_ENTRY(stage1_scores, Kv, Ptr, Array, Array, Array, Array, Array, I32, I32, Float, Ptr, Ptr, Ptr, Size, Ptr),
    SPECVLM_ENTRY(stage1_scores_layers, Kv, Ptr, Array, Array, Array, Array, Array, I32, I32, Float, Ptr, Ptr, Ptr, Size, I32, I32,
                  I32, Ptr),
    SPECVLM_ENTRY(select, Ptr, Array, Array, I32, Array, Array, Array, I32, Ptr, Ptr),
    SPECVLM_ENTRY(select_top_p, Ptr, Array, Array, I32, Array, Array, Array, I32, Ptr, Ptr, Ptr),
    SPECVLM_ENTRY(gather_kv, Kv, Ptr, Array, Array, Array, Array, I32, Kv, Ptr),
    SPECVLM_ENTRY(draft_decode_attn, Kv, Ptr, I32, I32, Float, Ptr, Ptr, Ptr, Size, Ptr),
    SPECVLM_ENTRY(verify_attn, Kv, Ptr, I32, I32, I32, Float, Ptr, Ptr, Ptr, Size, Ptr),
    SPECVLM_ENTRY(verify_tree_attn, Kv, Ptr, Ptr, I32, I32, I32, Float, Ptr, Ptr, Ptr, Size, Ptr),
    SPECVLM_ENTRY(accept, Ptr, Ptr, I32, I32, I32, Ptr, Ptr, Ptr, Ptr, Size),
    SPECVLM_ENTRY(accept_tree, Ptr, Ptr, Ptr, I32, I32, I32, Ptr, Ptr, Ptr, Ptr, Ptr, Size),
    SPECVLM_ENTRY(append_kv, Kv, Ptr, Ptr, I32, I32, Ptr, Ptr),
    SPECVLM_ENTRY(rollback_kv, Ptr, Ptr, I32, I32, Ptr),
    SPECVLM_ENTRY(compact_tree_kv, Kv, Ptr, Ptr, I32, I32, Ptr, Ptr),
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding() {
  g_data_ptr = PyUnicode_InternFromString("data_ptr");
  return g_data_ptr ? PyModule_Create(&g_module) : nullptr;
}
