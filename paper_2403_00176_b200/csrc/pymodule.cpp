// CPython module `_sod2calls`: the calls a program makes for every batch (bind, plan, run, output shapes, destroy), with
// their arguments taken straight from Python lists.  Through ctypes, building the argument arrays cost more than the
// calls themselves (the smallest fused group: 6 of 13 us a pass).  Marshalling only: every function hands its arguments
// to the C ABI of libsod2.so, releases the interpreter lock around it and returns its status.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <cstdint>
#include <new>

#include "../../include/sod2.h"

namespace {

// Small argument arrays live on the stack.  They start out as zeros: a missing address is a null address.
template <class T, int N>
struct Buf {
  T local[N] = {};
  T* p = local;
  bool reserve(Py_ssize_t n) {
    if (n <= N) return true;
    p = new (std::nothrow) T[n]();
    if (!p) { p = local; PyErr_NoMemory(); return false; }
    return true;
  }
  ~Buf() { if (p != local) delete[] p; }
};

bool as_i64(PyObject* o, int64_t* out) {
  if (PyLong_CheckExact(o)) {
    *out = PyLong_AsLongLong(o);
  } else {
    PyObject* l = PyNumber_Long(o);
    if (!l) return false;
    *out = PyLong_AsLongLong(l);
    Py_DECREF(l);
  }
  return !(*out == -1 && PyErr_Occurred());
}

bool as_ptr(PyObject* o, void** out) {
  if (o == Py_None) { *out = nullptr; return true; }
  *out = PyLong_AsVoidPtr(o);
  return !(*out == nullptr && PyErr_Occurred());
}
// An entry of a list of addresses may also be a ctypes.c_void_p.
bool as_entry(PyObject* o, void** out) {
  if (o == Py_None || PyLong_Check(o)) return as_ptr(o, out);
  PyObject* v = PyObject_GetAttrString(o, "value");
  if (!v) {
    PyErr_Format(PyExc_TypeError, "an address is wanted, got %.100s", Py_TYPE(o)->tp_name);
    return false;
  }
  const bool ok = as_ptr(v, out);
  Py_DECREF(v);
  return ok;
}

// At least `least` entries: what the list lacks is null, and refused by the call.
template <int N>
bool as_ptrs(PyObject* seq, Buf<void*, N>* out, Py_ssize_t least) {
  PyObject* f = PySequence_Fast(seq, "a sequence of addresses is wanted");
  if (!f) return false;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(f);
  bool ok = out->reserve(n > least ? n : least);
  for (Py_ssize_t i = 0; ok && i < n; ++i) ok = as_entry(PySequence_Fast_GET_ITEM(f, i), &out->p[i]);
  Py_DECREF(f);
  return ok;
}

bool want(Py_ssize_t got, Py_ssize_t n) {
  if (got == n) return true;
  PyErr_Format(PyExc_TypeError, "%zd arguments are wanted, got %zd", n, got);
  return false;
}

// bind(graph, names, rows) -> (status, binding)
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!want(n, 3)) return nullptr;
  void* g;
  if (!as_ptr(a[0], &g)) return nullptr;
  PyObject* names = PySequence_Fast(a[1], "a sequence of symbol names is wanted");
  if (!names) return nullptr;
  PyObject* rows = PySequence_Fast(a[2], "a sequence of rows is wanted");
  if (!rows) { Py_DECREF(names); return nullptr; }
  const Py_ssize_t n_sym = PySequence_Fast_GET_SIZE(names), n_req = PySequence_Fast_GET_SIZE(rows);
  Buf<const char*, 16> nm;
  Buf<int64_t, 128> val;
  bool ok = nm.reserve(n_sym) && val.reserve(n_sym * n_req);
  for (Py_ssize_t i = 0; ok && i < n_sym; ++i) ok = (nm.p[i] = PyUnicode_AsUTF8(PySequence_Fast_GET_ITEM(names, i))) != nullptr;
  for (Py_ssize_t r = 0; ok && r < n_req; ++r) {
    PyObject* row = PySequence_Fast(PySequence_Fast_GET_ITEM(rows, r), "a row of symbol values is wanted");
    if (!row) { ok = false; break; }
    if (PySequence_Fast_GET_SIZE(row) != n_sym) {
      PyErr_Format(PyExc_ValueError, "request %zd has %zd values for %zd symbols", r, PySequence_Fast_GET_SIZE(row), n_sym);
      ok = false;
    }
    for (Py_ssize_t i = 0; ok && i < n_sym; ++i) ok = as_i64(PySequence_Fast_GET_ITEM(row, i), &val.p[r * n_sym + i]);
    Py_DECREF(row);
  }
  PyObject* res = nullptr;
  if (ok) {
    sod2_binding* b = nullptr;
    int st;
    Py_BEGIN_ALLOW_THREADS
    st = sod2_bind_dims(static_cast<sod2_graph*>(g), static_cast<int>(n_req), static_cast<int>(n_sym), nm.p, val.p, &b);
    Py_END_ALLOW_THREADS
    res = Py_BuildValue("iN", st, PyLong_FromVoidPtr(b));
  }
  Py_DECREF(names);
  Py_DECREF(rows);
  return res;
}

// plan(graph, binding) -> (status, plan, arena bytes)
PyObject* py_plan(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void *g, *b;
  if (!want(n, 2) || !as_ptr(a[0], &g) || !as_ptr(a[1], &b)) return nullptr;
  sod2_plan_t* p = nullptr;
  size_t bytes = 0;
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = sod2_plan(static_cast<sod2_graph*>(g), static_cast<sod2_binding*>(b), &p, &bytes);
  Py_END_ALLOW_THREADS
  return Py_BuildValue("iNn", st, PyLong_FromVoidPtr(p), static_cast<Py_ssize_t>(bytes));
}

// run(how, plan, inputs, outputs, arena, arena bytes, stream, info) -> status; info: a writable buffer of sod2_run_info
PyObject* py_run(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (!want(n, 8)) return nullptr;
  int64_t how, bytes;
  void *p, *arena, *stream;
  Buf<void*, 64> in, out;
  int n_in = 0, n_out = 0;
  if (!as_i64(a[0], &how) || !as_ptr(a[1], &p)) return nullptr;
  sod2_plan_io_counts(static_cast<sod2_plan_t*>(p), &n_in, &n_out);
  if (!as_ptrs(a[2], &in, n_in) || !as_ptrs(a[3], &out, n_out) || !as_ptr(a[4], &arena) ||
      !as_i64(a[5], &bytes) || !as_ptr(a[6], &stream))
    return nullptr;
  Py_buffer info;
  if (PyObject_GetBuffer(a[7], &info, PyBUF_WRITABLE) != 0) return nullptr;
  if (info.len < static_cast<Py_ssize_t>(sizeof(sod2_run_info))) {
    PyBuffer_Release(&info);
    PyErr_SetString(PyExc_ValueError, "the run-info buffer is too small");
    return nullptr;
  }
  auto* fn = how == 0 ? sod2_run : how == 1 ? sod2_run_graph : sod2_run_exact;
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = fn(static_cast<sod2_plan_t*>(p), in.p, out.p, arena, static_cast<size_t>(bytes), stream, static_cast<sod2_run_info*>(info.buf));
  Py_END_ALLOW_THREADS
  PyBuffer_Release(&info);
  return PyLong_FromLong(st);
}

// output_shape(plan, arena, stream, request, output) -> list of extents, or the status if it is not 0
PyObject* py_output_shape(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void *p, *arena, *stream;
  int64_t r, o;
  if (!want(n, 5) || !as_ptr(a[0], &p) || !as_ptr(a[1], &arena) || !as_ptr(a[2], &stream) || !as_i64(a[3], &r) || !as_i64(a[4], &o)) return nullptr;
  int64_t dims[16];
  int rank = 0, st;
  Py_BEGIN_ALLOW_THREADS
  st = sod2_run_output_shape(static_cast<sod2_plan_t*>(p), arena, stream, static_cast<int>(r), static_cast<int>(o), dims, &rank);
  Py_END_ALLOW_THREADS
  if (st) return PyLong_FromLong(st);
  PyObject* l = PyList_New(rank);
  for (int i = 0; l && i < rank; ++i) PyList_SET_ITEM(l, i, PyLong_FromLongLong(dims[i]));
  return l;
}

PyObject* py_binding_destroy(PyObject*, PyObject* h) {
  void* p;
  if (!as_ptr(h, &p)) return nullptr;
  sod2_binding_destroy(static_cast<sod2_binding*>(p));
  Py_RETURN_NONE;
}
PyObject* py_plan_destroy(PyObject*, PyObject* h) {
  void* p;
  if (!as_ptr(h, &p)) return nullptr;
  Py_BEGIN_ALLOW_THREADS
  sod2_plan_destroy(static_cast<sod2_plan_t*>(p));
  Py_END_ALLOW_THREADS
  Py_RETURN_NONE;
}

#define FAST(f) reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(f))
PyMethodDef methods[] = {
    {"bind", FAST(py_bind), METH_FASTCALL, "sod2_bind_dims"},
    {"plan", FAST(py_plan), METH_FASTCALL, "sod2_plan"},
    {"run", FAST(py_run), METH_FASTCALL, "sod2_run (0), sod2_run_graph (1), sod2_run_exact (2)"},
    {"output_shape", FAST(py_output_shape), METH_FASTCALL, "sod2_run_output_shape"},
    {"binding_destroy", py_binding_destroy, METH_O, "sod2_binding_destroy"},
    {"plan_destroy", py_plan_destroy, METH_O, "sod2_plan_destroy"},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_sod2calls", "per-batch calls into libsod2.so", -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__sod2calls(void) { return PyModule_Create(&module); }
