// The per-layer calls of the Python binding, marshalled natively: kvswap_project_keys, kvswap_score_select and
// kvswap_sparse_decode take tensors and pass their addresses on, as binding.py's ctypes versions do, in whose place they
// are put.  A model that runs its own layers between the calls issues two of them per layer, and through ctypes a call
// cost 1.6 us of marshalling on top of 3.7 us of library and launch.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "kvswap.h"

namespace {

using ProjectFn = int (*)(const kvswap_shape*, const void*, const float*, void*, int32_t, int32_t, void*, size_t, void*);
using SelectFn = int (*)(const kvswap_shape*, const void*, const float*, const void*, int32_t*, int32_t*, float*, void*, size_t, void*);
using DecodeFn = int (*)(const kvswap_shape*, const void*, const void*, const void*, const int32_t*, const int32_t*, float*, float*,
                         void*, size_t, void*);

PyObject* g_resolve = nullptr;       // binding's callable: loads the library, returns what the calls need
PyObject* g_error = nullptr;         // KVSwapError
PyObject* g_shape = nullptr;         // kvswap_shape
PyObject* g_device = nullptr;        // () -> current device
PyObject* g_raw_stream = nullptr;    // (device) -> cudaStream_t of the current stream
ProjectFn g_project = nullptr;
SelectFn g_select = nullptr;
DecodeFn g_decode = nullptr;
PyObject *s_data_ptr, *s_numel, *s_element_size, *s_cuda_stream, *s_value;

bool ready() {
  if (g_decode != nullptr) return true;
  PyObject* t = PyObject_CallNoArgs(g_resolve);
  if (t == nullptr) return false;
  unsigned long long a, b, c;
  PyObject *device, *raw;
  if (!PyArg_ParseTuple(t, "KKKOO", &a, &b, &c, &device, &raw)) { Py_DECREF(t); return false; }
  g_device = Py_NewRef(device);
  g_raw_stream = Py_NewRef(raw);
  g_project = reinterpret_cast<ProjectFn>(a);
  g_select = reinterpret_cast<SelectFn>(b);
  g_decode = reinterpret_cast<DecodeFn>(c);
  Py_DECREF(t);
  return true;
}

bool as_u64(PyObject* o, unsigned long long* v) {      // steals o
  if (o == nullptr) return false;
  *v = PyLong_AsUnsignedLongLong(o);
  Py_DECREF(o);
  return !(*v == static_cast<unsigned long long>(-1) && PyErr_Occurred());
}

// Address of a tensor, NULL for None.
bool address(PyObject* t, void** p) {
  *p = nullptr;
  if (t == Py_None) return true;
  unsigned long long v;
  if (!as_u64(PyObject_CallMethodNoArgs(t, s_data_ptr), &v)) return false;
  *p = reinterpret_cast<void*>(v);
  return true;
}

bool size_of(PyObject* t, size_t* n) {
  *n = 0;
  if (t == Py_None) return true;
  unsigned long long a, b;
  if (!as_u64(PyObject_CallMethodNoArgs(t, s_numel), &a) || !as_u64(PyObject_CallMethodNoArgs(t, s_element_size), &b)) return false;
  *n = size_t(a) * size_t(b);
  return true;
}

// A torch stream, a handle (an int or a ctypes.c_void_p), or None: torch's current stream.
bool stream_of(PyObject* s, void** p) {
  *p = nullptr;
  PyObject* h;
  if (s == Py_None) {
    PyObject* dev = PyObject_CallNoArgs(g_device);
    if (dev == nullptr) return false;
    h = PyObject_CallOneArg(g_raw_stream, dev);
    Py_DECREF(dev);
  } else if (PyLong_Check(s)) {
    h = Py_NewRef(s);
  } else if ((h = PyObject_GetAttr(s, s_cuda_stream)) == nullptr && PyErr_ExceptionMatches(PyExc_AttributeError)) {
    PyErr_Clear();
    h = PyObject_GetAttr(s, s_value);
  }
  if (h == Py_None) { Py_DECREF(h); return true; }                  // the default stream
  unsigned long long v = 0;
  if (!as_u64(h, &v)) return false;
  *p = reinterpret_cast<void*>(v);
  return true;
}

bool int32_of(PyObject* o, int32_t* v) {
  PyObject* i = PyNumber_Long(o);
  if (i == nullptr) return false;
  const long long x = PyLong_AsLongLong(i);
  Py_DECREF(i);
  if (x == -1 && PyErr_Occurred()) return false;
  *v = int32_t(x);
  return true;
}

// Positional and keyword arguments into `out` by name; the last one, `stream`, defaults to None.
bool arguments(const char* fn, const char* const* names, int n, PyObject* const* args, Py_ssize_t n_pos, PyObject* kwnames, PyObject** out) {
  if (n_pos > n) { PyErr_Format(PyExc_TypeError, "%s() takes at most %d arguments (%zd given)", fn, n, n_pos); return false; }
  for (int i = 0; i < n; ++i) out[i] = i < n_pos ? args[i] : nullptr;
  const Py_ssize_t n_kw = kwnames ? PyTuple_GET_SIZE(kwnames) : 0;
  for (Py_ssize_t k = 0; k < n_kw; ++k) {
    int i = 0;
    while (i < n && PyUnicode_CompareWithASCIIString(PyTuple_GET_ITEM(kwnames, k), names[i]) != 0) ++i;
    if (i == n || out[i] != nullptr) {
      PyErr_Format(PyExc_TypeError, "%s() got an unexpected or repeated argument '%U'", fn, PyTuple_GET_ITEM(kwnames, k));
      return false;
    }
    out[i] = args[n_pos + k];
  }
  if (out[n - 1] == nullptr) out[n - 1] = Py_None;
  for (int i = 0; i < n; ++i)
    if (out[i] == nullptr) { PyErr_Format(PyExc_TypeError, "%s() missing argument '%s'", fn, names[i]); return false; }
  return true;
}

struct Shape {                        // the bytes of the ctypes structure
  Py_buffer view = {};
  bool get(PyObject* o) {
    const int is_shape = PyObject_IsInstance(o, g_shape);
    if (is_shape < 0) return false;
    if (is_shape == 0) { PyErr_Format(PyExc_TypeError, "shape: expected a kvswap_shape, got %.100s", Py_TYPE(o)->tp_name); return false; }
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) return false;
    if (view.len == Py_ssize_t(sizeof(kvswap_shape))) return true;
    PyErr_SetString(PyExc_TypeError, "shape: a kvswap_shape of another size");
    return false;
  }
  const kvswap_shape* ptr() const { return static_cast<const kvswap_shape*>(view.buf); }
  ~Shape() { if (view.obj != nullptr) PyBuffer_Release(&view); }
};

PyObject* done(int status, const char* where) {
  if (status == 0) Py_RETURN_NONE;
  PyObject* e = PyObject_CallFunction(g_error, "is", status, where);
  if (e != nullptr) { PyErr_SetObject(g_error, e); Py_DECREF(e); }
  return nullptr;
}

PyObject* project_keys(PyObject*, PyObject* const* args, Py_ssize_t n_pos, PyObject* kwnames) {
  static const char* const names[] = {"shape", "K", "proj", "meta_out", "n_begin", "n_end", "ws", "stream"};
  PyObject* a[8];
  Shape s;
  void *K, *proj, *meta, *ws, *st;
  int32_t n0, n1;
  size_t bytes;
  if (!ready() || !arguments("kvswap_project_keys", names, 8, args, n_pos, kwnames, a) || !s.get(a[0]) || !address(a[1], &K) ||
      !address(a[2], &proj) || !address(a[3], &meta) || !int32_of(a[4], &n0) || !int32_of(a[5], &n1) || !address(a[6], &ws) ||
      !size_of(a[6], &bytes) || !stream_of(a[7], &st))
    return nullptr;
  int status;
  Py_BEGIN_ALLOW_THREADS
  status = g_project(s.ptr(), K, static_cast<const float*>(proj), meta, n0, n1, ws, bytes, st);
  Py_END_ALLOW_THREADS
  return done(status, "kvswap_project_keys");
}

PyObject* score_select(PyObject*, PyObject* const* args, Py_ssize_t n_pos, PyObject* kwnames) {
  static const char* const names[] = {"shape", "q", "proj", "meta", "group_idx", "n_selected", "group_scores_opt", "ws", "stream"};
  PyObject* a[9];
  Shape s;
  void *q, *proj, *meta, *idx, *nsel, *scores, *ws, *st;
  size_t bytes;
  if (!ready() || !arguments("kvswap_score_select", names, 9, args, n_pos, kwnames, a) || !s.get(a[0]) || !address(a[1], &q) ||
      !address(a[2], &proj) || !address(a[3], &meta) || !address(a[4], &idx) || !address(a[5], &nsel) || !address(a[6], &scores) ||
      !address(a[7], &ws) || !size_of(a[7], &bytes) || !stream_of(a[8], &st))
    return nullptr;
  int status;
  Py_BEGIN_ALLOW_THREADS
  status = g_select(s.ptr(), q, static_cast<const float*>(proj), meta, static_cast<int32_t*>(idx), static_cast<int32_t*>(nsel),
                    static_cast<float*>(scores), ws, bytes, st);
  Py_END_ALLOW_THREADS
  return done(status, "kvswap_score_select");
}

PyObject* sparse_decode(PyObject*, PyObject* const* args, Py_ssize_t n_pos, PyObject* kwnames) {
  static const char* const names[] = {"shape", "q", "K", "V", "group_idx", "n_selected", "out", "lse_opt", "ws", "stream"};
  PyObject* a[10];
  Shape s;
  void *q, *K, *V, *idx, *nsel, *out, *lse, *ws, *st;
  size_t bytes;
  if (!ready() || !arguments("kvswap_sparse_decode", names, 10, args, n_pos, kwnames, a) || !s.get(a[0]) || !address(a[1], &q) ||
      !address(a[2], &K) || !address(a[3], &V) || !address(a[4], &idx) || !address(a[5], &nsel) || !address(a[6], &out) ||
      !address(a[7], &lse) || !address(a[8], &ws) || !size_of(a[8], &bytes) || !stream_of(a[9], &st))
    return nullptr;
  int status;
  Py_BEGIN_ALLOW_THREADS
  status = g_decode(s.ptr(), q, K, V, static_cast<const int32_t*>(idx), static_cast<const int32_t*>(nsel), static_cast<float*>(out),
                    static_cast<float*>(lse), ws, bytes, st);
  Py_END_ALLOW_THREADS
  return done(status, "kvswap_sparse_decode");
}

// setup(resolve, error, shape): resolve() -> (addresses of the three entry points, current-device and raw-stream
// callables); the classes KVSwapError and kvswap_shape.
PyObject* setup(PyObject*, PyObject* args) {
  PyObject *r, *e, *s;
  if (!PyArg_ParseTuple(args, "OOO", &r, &e, &s)) return nullptr;
  g_resolve = Py_NewRef(r);
  g_error = Py_NewRef(e);
  g_shape = Py_NewRef(s);
  Py_RETURN_NONE;
}

PyMethodDef kMethods[] = {
    {"setup", setup, METH_VARARGS, nullptr},
    {"kvswap_project_keys", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(project_keys)), METH_FASTCALL | METH_KEYWORDS,
     "kvswap_project_keys(shape, K, proj, meta_out, n_begin, n_end, ws, stream=None)\n--\n\nK_lr = Flatten(K) A for tokens n_begin <= n < n_end; ws may be None."},
    {"kvswap_score_select", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(score_select)), METH_FASTCALL | METH_KEYWORDS,
     "kvswap_score_select(shape, q, proj, meta, group_idx, n_selected, group_scores_opt, ws, stream=None)\n--\n\nLow-rank scores, group maxima and the indices of the top_k groups; group_scores_opt may be None."},
    {"kvswap_sparse_decode", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(sparse_decode)), METH_FASTCALL | METH_KEYWORDS,
     "kvswap_sparse_decode(shape, q, K, V, group_idx, n_selected, out, lse_opt, ws, stream=None)\n--\n\nAttention over the selected groups and the rolling-buffer tail; lse_opt may be None."},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_numel = PyUnicode_InternFromString("numel");
  s_element_size = PyUnicode_InternFromString("element_size");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  s_value = PyUnicode_InternFromString("value");
  return PyModule_Create(&kModule);
}
