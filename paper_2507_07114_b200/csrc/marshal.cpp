// The binding's calls into the library: tensors to pointers, lists of them to pointer tables, the current stream, the call.
// A step of a small bucket takes the GPU five microseconds; as Python and ctypes work its arguments took four (four workers)
// to eight (26) on the host, so that the host was what such a step waited for. Nothing is kept from one call for the next.
// What an argument is taken as is what ctypes takes it as. The arguments of a usual program are taken here; any other (a ctypes integer, a
// pointer object, ...) is a TypeError or OverflowError, nothing has been called then, and the binding leaves it to ctypes.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/PythonTorchFunctionTLS.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <array>
#include <exception>
#include <utility>
#include <vector>

namespace {

constexpr int kMaxArgs = 16, kMaxTables = 4, kTable = 64;
PyObject* g_data_ptr;   // "data_ptr"
PyObject* g_value;      // "value"
PyObject* g_pointer;    // ctypes.c_void_p

bool whole(PyObject* o, uint64_t* out) {   // modulo 2^64, as a C argument of that width takes an integer
  if (!PyLong_Check(o)) {
    PyErr_Format(PyExc_TypeError, "an integer is wanted, not %.100s", Py_TYPE(o)->tp_name);
    return false;
  }
  *out = PyLong_AsUnsignedLongLongMask(o);
  return !(*out == (uint64_t)-1 && PyErr_Occurred());
}

// A tensor's address (None: 0). Subclasses, modes that watch every call and other objects answer for themselves.
bool address(PyObject* o, bool plain, uint64_t* out) {
  if (o == Py_None) {
    *out = 0;
    return true;
  }
  if (plain && THPVariable_CheckExact(o)) {
    *out = reinterpret_cast<uint64_t>(THPVariable_Unpack(o).data_ptr());
    return true;
  }
  PyObject* r = PyObject_CallMethodNoArgs(o, g_data_ptr);
  if (!r) return false;
  *out = PyLong_Check(r) ? PyLong_AsUnsignedLongLong(r) : (PyErr_SetString(PyExc_TypeError, "data_ptr() is no integer"), 0);
  Py_DECREF(r);
  return !PyErr_Occurred();
}

bool handle(PyObject* o, uint64_t* out) {   // a ctypes.c_void_p, an integer or None
  if (o == Py_None) {
    *out = 0;
    return true;
  }
  if (PyLong_Check(o)) return whole(o, out);
  if (!PyObject_TypeCheck(o, reinterpret_cast<PyTypeObject*>(g_pointer))) {
    PyErr_Format(PyExc_TypeError, "a c_void_p, an integer or None is wanted, not %.100s", Py_TYPE(o)->tp_name);
    return false;
  }
  PyObject* v = PyObject_GetAttr(o, g_value);
  if (!v) return false;
  const bool ok = v == Py_None ? (*out = 0, true) : whole(v, out);
  Py_DECREF(v);
  return ok;
}

// Every argument of the library's functions that come here is a pointer or a 64-bit integer.
template <size_t... I>
int invoke(uint64_t fn, const uint64_t* a, std::index_sequence<I...>) {
  using Fn = int (*)(decltype((void)I, uint64_t{})...);
  return reinterpret_cast<Fn>(fn)(a[I]...);
}
template <size_t N>
int invoke_n(uint64_t fn, const uint64_t* a, size_t n) {
  if (n == N) return invoke(fn, a, std::make_index_sequence<N>{});
  if constexpr (N > 1) return invoke_n<N - 1>(fn, a, n);
  return -1;
}

struct Table {
  std::array<uint64_t, kTable> few;
  std::vector<uint64_t> many;
};

bool table(PyObject* o, bool plain, Table& t, uint64_t* out) {
  if (PyObject_Size(o) < 0) return false;      // (what is walked once has no length, and is no table)
  PyObject* seq = PySequence_Fast(o, "a sequence of tensors is wanted");
  if (!seq) return false;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
  uint64_t* p = t.few.data();
  bool ok = true;
  if (n > kTable) {
    t.many.assign((size_t)n, 0);
    p = t.many.data();
  } else {
    t.few.fill(0);      // (a table that is too short ends in null pointers)
  }
  for (Py_ssize_t i = 0; ok && i < n && i < PySequence_Fast_GET_SIZE(seq); ++i) {   // (an entry's own answer may change the list)
    PyObject* entry = PySequence_Fast_GET_ITEM(seq, i);
    Py_INCREF(entry);
    ok = address(entry, plain, &p[i]);
    Py_DECREF(entry);
  }
  Py_DECREF(seq);
  *out = reinterpret_cast<uint64_t>(p);
  return ok;
}

// call(function, kinds, context, *arguments) -> return code. Kinds, a letter per argument: u an integer, p a tensor or None, t a sequence
// of them, b bytes (a table made before), s nothing: the current stream goes there.
PyObject* call(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  if (nargs < 3) {
    PyErr_SetString(PyExc_TypeError, "call(function, kinds, context, ...)");
    return nullptr;
  }
  try {
    uint64_t fn = 0, a[kMaxArgs];
    Py_ssize_t klen = 0;
    const char* kinds = PyUnicode_AsUTF8AndSize(args[1], &klen);
    if (!kinds || !whole(args[0], &fn) || !handle(args[2], &a[0])) return nullptr;
    if (fn == 0 || klen + 1 > kMaxArgs) {
      PyErr_SetString(PyExc_ValueError, "no function, or too many arguments");
      return nullptr;
    }
    const bool plain = !at::impl::torch_function_mode_enabled();
    Table tables[kMaxTables];
    int used = 0;
    Py_ssize_t at = 3;
    for (Py_ssize_t k = 0; k < klen; ++k) {
      uint64_t* to = &a[k + 1];
      if (kinds[k] == 's') {
        *to = reinterpret_cast<uint64_t>(c10::cuda::getCurrentCUDAStream().stream());
        continue;
      }
      if (at >= nargs || (kinds[k] == 't' && used == kMaxTables)) {
        PyErr_SetString(PyExc_TypeError, "too few arguments, or too many tables");
        return nullptr;
      }
      PyObject* o = args[at++];
      bool ok;
      if (kinds[k] == 'p') ok = address(o, plain, to);
      else if (kinds[k] == 't') ok = table(o, plain, tables[used++], to);
      else if (kinds[k] == 'b') { char* b = PyBytes_AsString(o); ok = b != nullptr; *to = reinterpret_cast<uint64_t>(b); }
      else ok = whole(o, to);
      if (!ok) return nullptr;
    }
    if (at != nargs) {
      PyErr_SetString(PyExc_TypeError, "too many arguments");
      return nullptr;
    }
    int rc;
    Py_BEGIN_ALLOW_THREADS
    rc = invoke_n<kMaxArgs>(fn, a, (size_t)klen + 1);
    Py_END_ALLOW_THREADS
    return PyLong_FromLong(rc);
  } catch (const c10::Error& e) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what_without_backtrace());
  } catch (const std::exception& e) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
  } catch (...) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, "unknown C++ exception");
  }
  return nullptr;
}

PyMethodDef g_methods[] = {{"call", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(call)), METH_FASTCALL, "call(function, kinds, context, *arguments) -> return code"},
                           {nullptr, nullptr, 0, nullptr}};
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() {
  g_data_ptr = PyUnicode_InternFromString("data_ptr");
  g_value = PyUnicode_InternFromString("value");
  PyObject* ctypes = PyImport_ImportModule("ctypes");
  g_pointer = ctypes ? PyObject_GetAttrString(ctypes, "c_void_p") : nullptr;
  Py_XDECREF(ctypes);
  if (!g_data_ptr || !g_value || !g_pointer) return nullptr;
  return PyModule_Create(&g_module);
}
