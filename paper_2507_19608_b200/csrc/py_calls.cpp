// CPython entry points for the calls a serving loop makes once per layer and token
// (delta_attn_decode_step) or once per prompt (delta_state_reset, delta_attn_prefill, delta_state_view): argument marshalling for the C ABI
// of libdelta_attn.so without an interpreted line.  A decode step of one sequence takes 4 to 5 us on
// the device; in Python (six _ptr calls, torch.cuda.current_stream, a ctypes call of eleven
// converted arguments) its marshalling took 5 us on top of the launch itself, here 0.6 us.
// The library stays a plain C ABI: setup() receives the addresses of its functions.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

namespace {

typedef int (*decode_fn)(void*, const void*, const void*, const void*, void*, void*, void*, float, int32_t, void*);
typedef int (*prefill_fn)(void*, const void*, const void*, const void*, void*, int32_t, int32_t, int32_t, int32_t, float,
                          int32_t, void*);
typedef int (*reset_fn)(void*, void*);
typedef int (*view_fn)(const void*, int32_t, const void**, size_t*);

decode_fn g_decode;
prefill_fn g_prefill;
reset_fn g_reset;
view_fn g_view;
PyObject *g_ptr, *g_stream, *g_check, *g_make_view;   // the binding's _ptr, _stream, _check, _make_view
PyObject* g_streams;                                  // gives (current device, raw stream of a device), once torch is up
PyObject *g_get_device, *g_get_stream;                // those two
PyObject *s_data_ptr, *s_raw, *s_views, *s_detach, *s_decode, *s_prefill, *s_reset, *s_view;  // interned names

// Device (or host) address of a tensor, array, integer or None.
bool address(PyObject* o, void** out) {
  if (o == Py_None) { *out = nullptr; return true; }
  PyObject* v;
  if (PyLong_Check(o)) {
    v = Py_NewRef(o);
  } else {
    v = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!v) {
      if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return false;
      PyErr_Clear();
      v = PyObject_CallOneArg(g_ptr, o);              // numpy arrays; TypeError for the rest
      if (!v) return false;
      if (v == Py_None) { Py_DECREF(v); *out = nullptr; return true; }
    }
  }
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !(*out == nullptr && PyErr_Occurred());
}

// The stream argument: None stands for torch's current stream.
bool stream_of(PyObject* o, void** out) {
  PyObject* v;
  if (o == nullptr || o == Py_None) {
    if (!g_get_stream) {
      PyObject* pair = PyObject_CallNoArgs(g_streams);
      if (!pair) return false;
      PyObject *d, *s;
      const bool ok = PyArg_ParseTuple(pair, "OO", &d, &s);
      if (ok) { g_get_device = Py_NewRef(d); g_get_stream = Py_NewRef(s); }
      Py_DECREF(pair);
      if (!ok) return false;
    }
    PyObject* dev = PyObject_CallNoArgs(g_get_device);
    if (!dev) return false;
    v = PyObject_CallOneArg(g_get_stream, dev);
    Py_DECREF(dev);
  } else {
    v = PyObject_CallOneArg(g_stream, o);
  }
  if (!v) return false;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !(*out == nullptr && PyErr_Occurred());
}

// The library's state handle, kept as an integer on the Python state object.
bool handle_of(PyObject* st, void** out) {
  PyObject* v = PyObject_GetAttr(st, s_raw);
  if (!v) return false;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !(*out == nullptr && PyErr_Occurred());
}

bool int_of(PyObject* o, int32_t* out) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) return false;
  *out = (int32_t)v;
  return true;
}

// Positional and keyword arguments into slots[0..n); the last one (stream) may be missing, or as many
// are needed as `needed` says.
bool collect(const char* fn, const char* const* names, int n, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames,
             PyObject** slots, int needed = -1) {
  for (int i = 0; i < n; ++i) slots[i] = nullptr;
  if (nargs > n) {
    PyErr_Format(PyExc_TypeError, "%s() takes at most %d arguments (%zd given)", fn, n, nargs);
    return false;
  }
  for (Py_ssize_t i = 0; i < nargs; ++i) slots[i] = args[i];
  const Py_ssize_t nk = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
  for (Py_ssize_t k = 0; k < nk; ++k) {
    PyObject* name = PyTuple_GET_ITEM(kwnames, k);
    int at = -1;
    for (int i = 0; i < n; ++i)
      if (PyUnicode_CompareWithASCIIString(name, names[i]) == 0) at = i;
    if (at < 0 || slots[at]) {
      PyErr_Format(PyExc_TypeError, at < 0 ? "%s() got an unexpected keyword argument '%U'"
                                           : "%s() got multiple values for argument '%U'", fn, name);
      return false;
    }
    slots[at] = args[nargs + k];
  }
  for (int i = 0; i < (needed < 0 ? n - 1 : needed); ++i)
    if (!slots[i]) {
      PyErr_Format(PyExc_TypeError, "%s() missing required argument: '%s'", fn, names[i]);
      return false;
    }
  return true;
}

PyObject* finish(int status, PyObject* where) {
  if (status == 0) Py_RETURN_NONE;
  PyObject* s = PyLong_FromLong(status);
  if (!s) return nullptr;
  PyObject* argv[2] = {s, where};
  PyObject* r = PyObject_Vectorcall(g_check, argv, 2, nullptr);      // raises DeltaError
  Py_DECREF(s);
  return r;
}

PyObject* decode_step(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
  static const char* const names[] = {"st", "q_new", "k_new", "v_new", "k_cache", "v_cache", "out", "theta", "window", "stream"};
  PyObject* a[10];
  if (!collect("delta_attn_decode_step", names, 10, args, nargs, kwnames, a)) return nullptr;
  void *h, *p[6], *stream;
  if (!handle_of(a[0], &h)) return nullptr;
  for (int i = 0; i < 6; ++i)
    if (!address(a[1 + i], &p[i])) return nullptr;
  const double theta = PyFloat_AsDouble(a[7]);
  if (theta == -1.0 && PyErr_Occurred()) return nullptr;
  int32_t window;
  if (!int_of(a[8], &window) || !stream_of(a[9], &stream)) return nullptr;
  int status;
  Py_BEGIN_ALLOW_THREADS
  status = g_decode(h, p[0], p[1], p[2], p[3], p[4], p[5], (float)theta, window, stream);
  Py_END_ALLOW_THREADS
  return finish(status, s_decode);
}

PyObject* prefill(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
  static const char* const names[] = {"st", "q", "k", "v", "out", "T", "H", "H_kv", "d", "theta", "window", "stream"};
  PyObject* a[12];
  if (!collect("delta_attn_prefill", names, 12, args, nargs, kwnames, a)) return nullptr;
  void *h, *p[4], *stream;
  if (!handle_of(a[0], &h)) return nullptr;
  for (int i = 0; i < 4; ++i)
    if (!address(a[1 + i], &p[i])) return nullptr;
  int32_t v[4], window;
  for (int i = 0; i < 4; ++i)
    if (!int_of(a[5 + i], &v[i])) return nullptr;
  const double theta = PyFloat_AsDouble(a[9]);
  if (theta == -1.0 && PyErr_Occurred()) return nullptr;
  if (!int_of(a[10], &window) || !stream_of(a[11], &stream)) return nullptr;
  int status;
  Py_BEGIN_ALLOW_THREADS
  status = g_prefill(h, p[0], p[1], p[2], p[3], v[0], v[1], v[2], v[3], (float)theta, window, stream);
  Py_END_ALLOW_THREADS
  return finish(status, s_prefill);
}

PyObject* reset(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
  static const char* const names[] = {"st", "stream"};
  PyObject* a[2];
  if (!collect("delta_state_reset", names, 2, args, nargs, kwnames, a)) return nullptr;
  void *h, *stream = nullptr;                         // (host-side only: the library does not use the stream)
  if (!handle_of(a[0], &h)) return nullptr;
  if (a[1] && a[1] != Py_None && !stream_of(a[1], &stream)) return nullptr;
  return finish(g_reset(h, stream), s_reset);
}

// A tensor over one of the state's arrays: another one over the memory of the tensor kept in st.views, or a
// first one (the binding's _make_view).
PyObject* view(PyObject*, PyObject* const* args, Py_ssize_t nargs, PyObject* kwnames) {
  static const char* const names[] = {"st", "what"};
  PyObject* a[2];
  if (!collect("delta_state_view", names, 2, args, nargs, kwnames, a, 2)) return nullptr;
  void* h;
  int32_t what;
  if (!handle_of(a[0], &h) || !int_of(a[1], &what)) return nullptr;
  const void* p = nullptr;
  size_t n = 0;
  const int status = g_view(h, what, &p, &n);
  if (status != 0) return finish(status, s_view);
  PyObject* at = PyLong_FromVoidPtr((void*)p);
  PyObject* key = at ? PyTuple_Pack(2, a[1], at) : nullptr;
  PyObject* views = key ? PyObject_GetAttr(a[0], s_views) : nullptr;
  PyObject* t = nullptr;
  if (views && PyDict_Check(views)) t = Py_XNewRef(PyDict_GetItemWithError(views, key));
  if (views && !t && !PyErr_Occurred()) {
    PyObject* size = PyLong_FromSize_t(n);
    PyObject* argv[4] = {a[0], a[1], at, size};
    if (size) t = PyObject_Vectorcall(g_make_view, argv, 4, nullptr);
    Py_XDECREF(size);
  }
  PyObject* r = t ? PyObject_CallMethodNoArgs(t, s_detach) : nullptr;
  Py_XDECREF(t);
  Py_XDECREF(views);
  Py_XDECREF(key);
  Py_XDECREF(at);
  return r;
}

// setup(addresses of decode, prefill, reset, view, _ptr, _stream, _check, _torch_streams, _make_view)
PyObject* setup(PyObject*, PyObject* args) {
  unsigned long long f[4];
  PyObject* o[5];
  if (!PyArg_ParseTuple(args, "KKKKOOOOO", &f[0], &f[1], &f[2], &f[3], &o[0], &o[1], &o[2], &o[3], &o[4])) return nullptr;
  g_decode = (decode_fn)(uintptr_t)f[0];
  g_prefill = (prefill_fn)(uintptr_t)f[1];
  g_reset = (reset_fn)(uintptr_t)f[2];
  g_view = (view_fn)(uintptr_t)f[3];
  PyObject** to[5] = {&g_ptr, &g_stream, &g_check, &g_streams, &g_make_view};
  for (int i = 0; i < 5; ++i) { Py_XDECREF(*to[i]); *to[i] = Py_NewRef(o[i]); }
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"setup", setup, METH_VARARGS, nullptr},
    {"delta_attn_decode_step", (PyCFunction)(void (*)(void))decode_step, METH_FASTCALL | METH_KEYWORDS, nullptr},
    {"delta_attn_prefill", (PyCFunction)(void (*)(void))prefill, METH_FASTCALL | METH_KEYWORDS, nullptr},
    {"delta_state_reset", (PyCFunction)(void (*)(void))reset, METH_FASTCALL | METH_KEYWORDS, nullptr},
    {"delta_state_view", (PyCFunction)(void (*)(void))view, METH_FASTCALL | METH_KEYWORDS, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_raw = PyUnicode_InternFromString("raw");
  s_decode = PyUnicode_InternFromString("delta_attn_decode_step");
  s_prefill = PyUnicode_InternFromString("delta_attn_prefill");
  s_reset = PyUnicode_InternFromString("delta_state_reset");
  s_view = PyUnicode_InternFromString("delta_state_view");
  s_views = PyUnicode_InternFromString("views");
  s_detach = PyUnicode_InternFromString("detach");
  return PyModule_Create(&module);
}
