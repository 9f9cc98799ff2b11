// The calls of the Python binding whose host work is many small objects, as a CPython module: a verdict comes back as some
// thirty arrays in dictionaries, an upload goes out as nine. Through ctypes and numpy's Python interface that work took about
// as long as the call itself (a verdict of a small job: 24 us, 13 of them in the library; an upload of 8,000 records: 34 us);
// here an array is one allocation. Everything else of the binding stays in Python.
//
// The module has no copy of the library: setup() is given the addresses of the functions it calls.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#define NPY_NO_DEPRECATED_API NPY_1_7_API_VERSION
#include <numpy/arrayobject.h>
#include <cstring>
#include <vector>
#include "../../include/ccld.h"

namespace {

decltype(&ccld_get_verdict_columns) f_verdict = nullptr;
decltype(&ccld_trace_upload) f_upload = nullptr;
decltype(&ccld_take_optable) f_optable = nullptr;
decltype(&ccld_take_rank_stats) f_stats = nullptr;
decltype(&ccld_host_release) f_release = nullptr;

struct Column { PyObject* name; int type; Py_ssize_t at; };            // at: bytes of an entry before the column
struct Plan { std::vector<Column> cols; Py_ssize_t size = 0; };        // in the order of the dictionary; size: bytes of an entry
Plan p_rows, p_alerts, p_suspects;
PyObject* n_verdict[15]; PyObject *n_rc, *n_comm_rows, *n_alerts, *n_suspects;
PyObject* n_upload[9];
constexpr Py_ssize_t UPLOAD_SIZE[9] = {4, 4, 4, 1, 8, 8, 8, 4, 4};

// A one-dimensional array of n entries at p, kept alive by owner.
PyObject* view_of(PyObject* owner, void* p, Py_ssize_t n, int type) {
  npy_intp dim = n;
  PyObject* a = PyArray_New(&PyArray_Type, 1, &dim, type, nullptr, n ? p : nullptr, 0, n ? NPY_ARRAY_CARRAY : 0, nullptr);
  if (!a || !n) return a;
  Py_INCREF(owner);
  if (PyArray_SetBaseObject((PyArrayObject*)a, owner) < 0) { Py_DECREF(a); return nullptr; }
  return a;
}
bool put(PyObject* dict, PyObject* key, PyObject* value) {             // takes the reference
  if (!value) return false;
  const int r = PyDict_SetItem(dict, key, value);
  Py_DECREF(value);
  return r == 0;
}
bool put(PyObject* dict, const char* key, PyObject* value) {
  if (!value) return false;
  const int r = PyDict_SetItemString(dict, key, value);
  Py_DECREF(value);
  return r == 0;
}

// A list of n entries that the library holds column by column, as one array per field (the first `cap` entries), in memory of
// its own: the library's area serves the next call.
PyObject* take(const void* src, Py_ssize_t n, Py_ssize_t cap, const Plan& plan) {
  PyObject* out = PyDict_New();
  if (!out) return nullptr;
  PyObject* buf = nullptr;
  char* p = nullptr;
  if (n) {
    npy_intp bytes = n * plan.size;
    buf = PyArray_SimpleNew(1, &bytes, NPY_UINT8);
    if (!buf) { Py_DECREF(out); return nullptr; }
    p = (char*)PyArray_DATA((PyArrayObject*)buf);
    std::memcpy(p, src, (size_t)bytes);
  }
  bool ok = true;
  for (const Column& c : plan.cols) if (ok) ok = put(out, c.name, view_of(buf, p + c.at * n, n < cap ? n : cap, c.type));
  Py_XDECREF(buf);
  if (!ok) { Py_DECREF(out); return nullptr; }
  return out;
}

// A pinned block of the library, given back once no array refers to it any more.
void release_block(PyObject* capsule) {
  ccld_host_block* b = (ccld_host_block*)PyCapsule_GetPointer(capsule, "ccld_host_block");
  if (b) { f_release(b); delete b; }
}
PyObject* own_block(const ccld_host_block& block) {
  ccld_host_block* b = new ccld_host_block(block);
  PyObject* c = PyCapsule_New(b, "ccld_host_block", release_block);
  if (!c) { f_release(b); delete b; }
  return c;
}

int typenum(char kind, long size) {
  switch (kind) {
    case 'f': return NPY_FLOAT64;
    case 'i': return size == 8 ? NPY_INT64 : NPY_INT32;
    default: return size == 8 ? NPY_UINT64 : NPY_UINT32;
  }
}

bool read_plan(PyObject* seq, Plan& plan) {                            // ((name, kind, bytes, at), ...)
  plan.cols.clear(); plan.size = 0;
  const Py_ssize_t n = PyTuple_Size(seq);
  for (Py_ssize_t i = 0; i < n; ++i) {
    PyObject* name; const char* kind; long size; Py_ssize_t at;
    if (!PyArg_ParseTuple(PyTuple_GET_ITEM(seq, i), "Osln", &name, &kind, &size, &at)) return false;
    Py_INCREF(name);
    plan.cols.push_back(Column{name, typenum(kind[0], size), at});
    plan.size += size;
  }
  return n >= 0;
}
bool read_names(PyObject* seq, PyObject** to, Py_ssize_t n) {
  if (PyTuple_Size(seq) != n) { PyErr_SetString(PyExc_ValueError, "wrong number of names"); return false; }
  for (Py_ssize_t i = 0; i < n; ++i) { to[i] = PyTuple_GET_ITEM(seq, i); Py_INCREF(to[i]); }
  return true;
}

// setup(addresses, verdict names, upload names, rows, alerts, suspects)
PyObject* setup(PyObject*, PyObject* args) {
  unsigned long long a[5];
  PyObject *v, *u, *r, *al, *s;
  if (!PyArg_ParseTuple(args, "(KKKKK)O!O!O!O!O!", &a[0], &a[1], &a[2], &a[3], &a[4], &PyTuple_Type, &v, &PyTuple_Type, &u,
                        &PyTuple_Type, &r, &PyTuple_Type, &al, &PyTuple_Type, &s)) return nullptr;
  if (!read_names(v, n_verdict, 15) || !read_names(u, n_upload, 9) || !read_plan(r, p_rows) || !read_plan(al, p_alerts) || !read_plan(s, p_suspects)) return nullptr;
  f_verdict = (decltype(f_verdict))a[0]; f_upload = (decltype(f_upload))a[1]; f_optable = (decltype(f_optable))a[2];
  f_stats = (decltype(f_stats))a[3]; f_release = (decltype(f_release))a[4];
  n_rc = PyUnicode_InternFromString("rc"); n_comm_rows = PyUnicode_InternFromString("comm_rows");
  n_alerts = PyUnicode_InternFromString("alerts"); n_suspects = PyUnicode_InternFromString("suspects");
  Py_RETURN_NONE;
}

// verdict(context, window, rows_cap, alerts_cap, suspects_cap) -> dictionary with the return code under "rc"
PyObject* verdict(PyObject*, PyObject* args) {
  unsigned long long h; unsigned int window; Py_ssize_t cap[3];
  if (!PyArg_ParseTuple(args, "KInnn", &h, &window, &cap[0], &cap[1], &cap[2])) return nullptr;
  for (Py_ssize_t& c : cap) if (c < 0) c = 0;
  ccld_verdict v; ccld_verdict_columns c;
  std::memset(&v, 0, sizeof v); std::memset(&c, 0, sizeof c);
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_verdict((ccld_ctx*)h, window, &v, &c);
  Py_END_ALLOW_THREADS
  PyObject* out = PyDict_New();
  if (!out) return nullptr;
  const unsigned long long n[15] = {v.n_records, v.n_groups, v.n_slots, v.n_rejected, v.n_complete, v.n_incomplete, v.n_barrier, v.n_analysed,
                                    v.n_flag_skew, v.n_flag_dur, v.n_opset_mismatch, v.error_bits, v.n_comm_rows_total, v.n_alerts_total, v.n_suspects_total};
  bool ok = true;
  for (int i = 0; i < 15 && ok; ++i) ok = put(out, n_verdict[i], PyLong_FromUnsignedLongLong(n[i]));
  ok = ok && put(out, n_rc, PyLong_FromLong(rc)) && put(out, n_comm_rows, take(c.rows, c.n_rows, cap[0], p_rows)) &&
       put(out, n_alerts, take(c.alerts, c.n_alerts, cap[1], p_alerts)) && put(out, n_suspects, take(c.suspects, c.n_suspects, cap[2], p_suspects));
  if (!ok) { Py_DECREF(out); return nullptr; }
  return out;
}

// upload(context, window, columns) -> (return code, arrays to keep), or None where a column is not a plain numpy array of the
// column's size: the general way is Python's then
PyObject* upload(PyObject*, PyObject* args) {
  unsigned long long h; unsigned int window; PyObject* cols;
  if (!PyArg_ParseTuple(args, "KIO!", &h, &window, &PyDict_Type, &cols)) return nullptr;
  const void* p[9]; unsigned long long n = 0;
  PyObject* keep[9]; Py_ssize_t n_keep = 0;
  for (int i = 0; i < 9; ++i) {
    PyObject* a = PyDict_GetItemWithError(cols, n_upload[i]);
    if (!a && PyErr_Occurred()) return nullptr;
    p[i] = nullptr;
    if (!a || a == Py_None) continue;
    if (!PyArray_CheckExact(a) || PyArray_ITEMSIZE((PyArrayObject*)a) != UPLOAD_SIZE[i] || !PyArray_IS_C_CONTIGUOUS((PyArrayObject*)a)) Py_RETURN_NONE;
    const unsigned long long m = (unsigned long long)PyArray_SIZE((PyArrayObject*)a);
    if (m) p[i] = PyArray_DATA((PyArrayObject*)a);
    if (i == 0) n = m;
    keep[n_keep++] = a;
  }
  if (!n_keep) Py_RETURN_NONE;
  PyObject* held = PyTuple_New(n_keep);
  if (!held) return nullptr;
  for (Py_ssize_t i = 0; i < n_keep; ++i) { Py_INCREF(keep[i]); PyTuple_SET_ITEM(held, i, keep[i]); }
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_upload((ccld_ctx*)h, window, n, 0, (const uint32_t*)p[0], (const uint32_t*)p[1], (const uint32_t*)p[2], (const uint8_t*)p[3],
                (const uint64_t*)p[4], (const int64_t*)p[5], (const int64_t*)p[6], (const uint32_t*)p[7], (const uint32_t*)p[8],
                0, nullptr, nullptr, nullptr, 0, nullptr);
  Py_END_ALLOW_THREADS
  return Py_BuildValue("(iN)", rc, held);
}

// rank_stats(context, ranks) -> (return code, dictionary or None); the arrays share a pinned block
PyObject* rank_stats(PyObject*, PyObject* args) {
  unsigned long long h; unsigned int n;
  if (!PyArg_ParseTuple(args, "KI", &h, &n)) return nullptr;
  ccld_host_rank_stats s;
  std::memset(&s, 0, sizeof s);
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_stats((ccld_ctx*)h, n, &s);
  Py_END_ALLOW_THREADS
  if (rc != CCLD_OK) return Py_BuildValue("(iO)", rc, Py_None);
  PyObject* own = own_block(s.block);
  if (!own) return nullptr;
  PyObject* out = PyDict_New();
  npy_intp dims[2] = {(npy_intp)n, 4};
  PyObject* votes = out ? PyArray_New(&PyArray_Type, 2, dims, NPY_UINT32, nullptr, n ? (void*)s.votes : nullptr, 0, n ? NPY_ARRAY_CARRAY : 0, nullptr) : nullptr;
  bool ok = votes != nullptr;
  if (ok && n) { Py_INCREF(own); ok = PyArray_SetBaseObject((PyArrayObject*)votes, own) == 0; }
  if (!ok) Py_XDECREF(votes);
  ok = ok && put(out, "votes", votes) && put(out, "ops", view_of(own, (void*)s.ops, n, NPY_UINT32)) &&
       put(out, "bw_cnt", view_of(own, (void*)s.bw_cnt, n, NPY_UINT32)) && put(out, "bw_sum", view_of(own, (void*)s.bw_sum, n, NPY_FLOAT64));
  Py_DECREF(own);
  if (!ok) { Py_XDECREF(out); return nullptr; }
  return Py_BuildValue("(iN)", rc, out);
}

// optable(context, window) -> (return code, dictionary or None); the arrays share a pinned block
PyObject* optable(PyObject*, PyObject* args) {
  unsigned long long h; unsigned int window;
  if (!PyArg_ParseTuple(args, "KI", &h, &window)) return nullptr;
  ccld_host_optable x;
  std::memset(&x, 0, sizeof x);
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_optable((ccld_ctx*)h, window, &x);
  Py_END_ALLOW_THREADS
  if (rc != CCLD_OK) return Py_BuildValue("(iO)", rc, Py_None);
  PyObject* own = own_block(x.block);
  if (!own) return nullptr;
  PyObject* out = PyDict_New();
  if (!out) { Py_DECREF(own); return nullptr; }
  const ccld_optable& t = x.t;
  const Py_ssize_t G = (Py_ssize_t)t.n_groups, S = (Py_ssize_t)t.n_slots;
  const struct { const char* name; const void* p; Py_ssize_t n; int type; } cols[] = {
      {"e_min", t.e_min, G, NPY_INT64}, {"arrival_skew", t.arrival_skew, G, NPY_INT64}, {"t_max", t.t_max, G, NPY_INT64}, {"t_min", t.t_min, G, NPY_INT64},
      {"span", t.span, G, NPY_INT64}, {"med_skew", t.med_skew, G, NPY_INT64}, {"mad_skew", t.mad_skew, G, NPY_INT64}, {"med_dur", t.med_dur, G, NPY_INT64},
      {"mad_dur", t.mad_dur, G, NPY_INT64}, {"rank_tmin", t.rank_tmin, G, NPY_UINT32}, {"rank_tmax", t.rank_tmax, G, NPY_UINT32},
      {"max_chg", t.max_chg, G, NPY_UINT32}, {"rank_max_chg", t.rank_max_chg, G, NPY_UINT32}, {"n_present", t.n_present, G, NPY_UINT32},
      {"gflags", t.gflags, G, NPY_UINT32}, {"busbw", t.busbw, G, NPY_FLOAT64}, {"flags", t.flags, S, NPY_UINT8}, {"perm", t.perm, S, NPY_UINT32},
      {"comm", x.comm, G, NPY_UINT32}, {"seq", x.seq, G, NPY_UINT32}, {"slot0", x.slot0, G, NPY_UINT64}};
  bool ok = put(out, "n_groups", PyLong_FromSsize_t(G)) && put(out, "n_slots", PyLong_FromSsize_t(S));
  for (const auto& c : cols) ok = ok && put(out, c.name, view_of(own, const_cast<void*>(c.p), c.n, c.type));
  Py_DECREF(own);
  if (!ok) { Py_DECREF(out); return nullptr; }
  return Py_BuildValue("(iN)", rc, out);
}

PyMethodDef methods[] = {{"setup", setup, METH_VARARGS, "Addresses of the library's functions, names of fields."},
                         {"verdict", verdict, METH_VARARGS, "ccld_get_verdict_columns as a dictionary of arrays."},
                         {"upload", upload, METH_VARARGS, "ccld_trace_upload of numpy columns."},
                         {"rank_stats", rank_stats, METH_VARARGS, "ccld_take_rank_stats as a dictionary of arrays."},
                         {"optable", optable, METH_VARARGS, "ccld_take_optable as a dictionary of arrays."},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) {
  import_array();
  return PyModule_Create(&module);
}
