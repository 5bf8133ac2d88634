// CPython front end of the C ABI for the calls of a user's inner loop: marshals torch tensors (used purely as memory
// handles) and numbers into the C call.  Small problems are bound by the host: through ctypes with torch's stream object
// a call spent 5-6 us in Python before the first launch, here about 1 us.  No arithmetic, no torch headers: tensors are
// asked for data_ptr() and nbytes, the current stream for its raw handle.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include <tuple>
#include <utility>

#include "../../include/mxattn.h"

namespace {

PyObject *g_data_ptr, *g_nbytes;              // interned method / attribute names
PyObject *g_get_device, *g_get_stream;        // torch._C._cuda_getDevice, torch._C._cuda_getCurrentRawStream

struct Args {
  PyObject* const* a;
  Py_ssize_t n, i = 0;
  bool ok = true;
  PyObject* tensor = nullptr;                 // the tensor read last (a size_t parameter is its size in bytes)
  PyObject* next() {
    if (i < n) return a[i++];
    if (ok) PyErr_SetString(PyExc_TypeError, "too few arguments");
    ok = false;
    return nullptr;
  }
};

// the value of a Python call's result as an unsigned 64-bit number (steals the reference)
uint64_t take_u64(Args& x, PyObject* r) {
  if (!r) { x.ok = false; return 0; }
  const uint64_t v = PyLong_AsUnsignedLongLong(r);
  Py_DECREF(r);
  if (v == (uint64_t)-1 && PyErr_Occurred()) x.ok = false;
  return v;
}

template <typename T> struct Get;
template <> struct Get<const void*> {
  static const void* from(Args& x) {
    PyObject* o = x.next();
    if (!x.ok) return nullptr;
    x.tensor = o;
    if (o == Py_None) return nullptr;
    return (const void*)take_u64(x, PyObject_CallMethodNoArgs(o, g_data_ptr));
  }
};
template <> struct Get<void*> { static void* from(Args& x) { return (void*)Get<const void*>::from(x); } };
template <> struct Get<size_t> {
  static size_t from(Args& x) {
    if (!x.ok || !x.tensor || x.tensor == Py_None) return 0;
    return (size_t)take_u64(x, PyObject_GetAttr(x.tensor, g_nbytes));
  }
};
template <> struct Get<int64_t> {
  static int64_t from(Args& x) {
    PyObject* o = x.next();
    if (!x.ok) return 0;
    const long long v = PyLong_AsLongLong(o);
    if (v == -1 && PyErr_Occurred()) x.ok = false;
    return v;
  }
};
template <> struct Get<int> {
  static int from(Args& x) {
    const int64_t v = Get<int64_t>::from(x);
    if (x.ok && v != (int)v) { PyErr_SetString(PyExc_OverflowError, "int out of range"); x.ok = false; }
    return (int)v;
  }
};
template <> struct Get<unsigned> {
  static unsigned from(Args& x) { return (unsigned)Get<int64_t>::from(x); }
};
template <> struct Get<float> {
  static float from(Args& x) {
    PyObject* o = x.next();
    if (!x.ok) return 0.0f;
    const double v = PyFloat_AsDouble(o);
    if (v == -1.0 && PyErr_Occurred()) x.ok = false;
    return (float)v;
  }
};

void* current_stream(Args& x) {
  if (!x.ok) return nullptr;
  PyObject* dev = PyObject_CallNoArgs(g_get_device);
  if (!dev) { x.ok = false; return nullptr; }
  PyObject* s = PyObject_CallOneArg(g_get_stream, dev);
  Py_DECREF(dev);
  return (void*)take_u64(x, s);
}

template <size_t I, typename T> void fill_one(T& v, Args& x) {
  using E = std::tuple_element_t<I, T>;
  if constexpr (I + 1 == std::tuple_size_v<T>) std::get<I>(v) = current_stream(x);
  else std::get<I>(v) = Get<E>::from(x);
}
template <typename T, size_t... I> void fill(T& v, Args& x, std::index_sequence<I...>) { (fill_one<I>(v, x), ...); }

// fn's parameters come from the Python arguments in order (a tensor gives a pointer; a size_t is the size in bytes of the
// tensor before it); the last one is torch's current stream.  Returns the status as a Python int.
template <typename... A>
PyObject* invoke(int (*fn)(A...), PyObject* const* args, Py_ssize_t nargs) {
  Args x{args, nargs};
  std::tuple<A...> v;
  fill(v, x, std::index_sequence_for<A...>{});
  if (x.ok && x.i != nargs) { PyErr_SetString(PyExc_TypeError, "too many arguments"); x.ok = false; }
  if (!x.ok) return nullptr;
  int rc;
  Py_BEGIN_ALLOW_THREADS                       // as through ctypes: other threads run while the call enqueues (or waits)
  rc = std::apply(fn, v);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

#define CALL(name) \
  PyObject* py_##name(PyObject*, PyObject* const* args, Py_ssize_t nargs) { return invoke(mxattn_##name, args, nargs); }
CALL(quantize_mxfp4) CALL(quantize_mxfp4_batched) CALL(quantize_mxfp4_qmax) CALL(tensor_amax) CALL(quantize_nvfp4)
CALL(forward) CALL(forward_static) CALL(forward_ws) CALL(forward_prequantized) CALL(forward_bf16) CALL(forward_nvfp4)
CALL(forward_host) CALL(rowsum_diagnostic)
#undef CALL

PyObject* py_init(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
  if (nargs != 2) { PyErr_SetString(PyExc_TypeError, "init(get_device, get_raw_stream)"); return nullptr; }
  Py_XDECREF(g_get_device); Py_XDECREF(g_get_stream);
  g_get_device = Py_NewRef(args[0]);
  g_get_stream = Py_NewRef(args[1]);
  Py_RETURN_NONE;
}

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, nullptr}
PyMethodDef g_methods[] = {
    ENTRY(init), ENTRY(quantize_mxfp4), ENTRY(quantize_mxfp4_batched), ENTRY(quantize_mxfp4_qmax), ENTRY(tensor_amax),
    ENTRY(quantize_nvfp4), ENTRY(forward), ENTRY(forward_static), ENTRY(forward_ws), ENTRY(forward_prequantized),
    ENTRY(forward_bf16), ENTRY(forward_nvfp4), ENTRY(forward_host), ENTRY(rowsum_diagnostic), {nullptr, nullptr, 0, nullptr}};
#undef ENTRY
PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_mxcall", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__mxcall(void) {
  g_data_ptr = PyUnicode_InternFromString("data_ptr");
  g_nbytes = PyUnicode_InternFromString("nbytes");
  return (g_data_ptr && g_nbytes) ? PyModule_Create(&g_module) : nullptr;
}
