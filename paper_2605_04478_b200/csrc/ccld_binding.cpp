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
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>
#include "../../include/ccld.h"

namespace {

decltype(&ccld_get_verdict_columns) f_verdict = nullptr;
decltype(&ccld_trace_upload) f_upload = nullptr;
decltype(&ccld_take_optable) f_optable = nullptr;
decltype(&ccld_take_rank_stats) f_stats = nullptr;
decltype(&ccld_host_release) f_release = nullptr;
decltype(&ccld_get_optable) f_table = nullptr;
decltype(&ccld_locate_hang) f_hang = nullptr;
decltype(&ccld_locate_hangs) f_hangs = nullptr;
decltype(&ccld_opset_check) f_opset = nullptr;
decltype(&ccld_derive_rates) f_rates = nullptr;
decltype(&ccld_get_ranges) f_ranges = nullptr;

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
  ccld_host_block* b = new (std::nothrow) ccld_host_block(block);
  if (!b) { ccld_host_block gone = block; f_release(&gone); return PyErr_NoMemory(); }
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
  unsigned long long a[11];
  PyObject *v, *u, *r, *al, *s;
  if (!PyArg_ParseTuple(args, "(KKKKKKKKKKK)O!O!O!O!O!", &a[0], &a[1], &a[2], &a[3], &a[4], &a[5], &a[6], &a[7], &a[8], &a[9], &a[10], &PyTuple_Type, &v, &PyTuple_Type, &u,
                        &PyTuple_Type, &r, &PyTuple_Type, &al, &PyTuple_Type, &s)) return nullptr;
  if (!read_names(v, n_verdict, 15) || !read_names(u, n_upload, 9) || !read_plan(r, p_rows) || !read_plan(al, p_alerts) || !read_plan(s, p_suspects)) return nullptr;
  f_verdict = (decltype(f_verdict))a[0]; f_upload = (decltype(f_upload))a[1]; f_optable = (decltype(f_optable))a[2];
  f_stats = (decltype(f_stats))a[3]; f_release = (decltype(f_release))a[4];
  f_table = (decltype(f_table))a[5]; f_hang = (decltype(f_hang))a[6]; f_hangs = (decltype(f_hangs))a[7]; f_opset = (decltype(f_opset))a[8];
  f_rates = (decltype(f_rates))a[9]; f_ranges = (decltype(f_ranges))a[10];
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
// column's size, or the ranks, whose number is the window's, are not there: the general way is Python's then
PyObject* upload(PyObject*, PyObject* args) {
  unsigned long long h; unsigned int window; PyObject* cols;
  if (!PyArg_ParseTuple(args, "KIO!", &h, &window, &PyDict_Type, &cols)) return nullptr;
  const void* p[9]; unsigned long long n = 0;
  PyObject* keep[9]; Py_ssize_t n_keep = 0;
  for (int i = 0; i < 9; ++i) {
    PyObject* a = PyDict_GetItemWithError(cols, n_upload[i]);
    if (!a && PyErr_Occurred()) return nullptr;
    p[i] = nullptr;
    if (!a || a == Py_None) { if (i == 0) Py_RETURN_NONE; continue; }
    if (!PyArray_CheckExact(a) || PyArray_ITEMSIZE((PyArrayObject*)a) != UPLOAD_SIZE[i] || !PyArray_IS_C_CONTIGUOUS((PyArrayObject*)a) ||
        PyDataType_REFCHK(PyArray_DESCR((PyArrayObject*)a))) Py_RETURN_NONE;      // (references to objects have eight bytes too)
    const unsigned long long m = (unsigned long long)PyArray_SIZE((PyArrayObject*)a);
    if (m) p[i] = PyArray_DATA((PyArrayObject*)a);
    if (i == 0) n = m;
    keep[n_keep++] = a;
  }
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

// table(context, window) -> (return code, dictionary of counts and device addresses); a null address is None
PyObject* table(PyObject*, PyObject* args) {
  unsigned long long h; unsigned int window;
  if (!PyArg_ParseTuple(args, "KI", &h, &window)) return nullptr;
  ccld_optable t;
  std::memset(&t, 0, sizeof t);
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_table((ccld_ctx*)h, window, &t);
  Py_END_ALLOW_THREADS
  PyObject* out = PyDict_New();
  if (!out) return nullptr;
  const struct { const char* name; const void* p; } cols[] = {
      {"e_min", t.e_min}, {"arrival_skew", t.arrival_skew}, {"t_max", t.t_max}, {"t_min", t.t_min}, {"span", t.span}, {"med_skew", t.med_skew},
      {"mad_skew", t.mad_skew}, {"med_dur", t.med_dur}, {"mad_dur", t.mad_dur}, {"rank_tmin", t.rank_tmin}, {"rank_tmax", t.rank_tmax},
      {"max_chg", t.max_chg}, {"rank_max_chg", t.rank_max_chg}, {"n_present", t.n_present}, {"gflags", t.gflags}, {"busbw", t.busbw},
      {"flags", t.flags}, {"perm", t.perm}};
  bool ok = put(out, "n_groups", PyLong_FromUnsignedLongLong(t.n_groups)) && put(out, "n_slots", PyLong_FromUnsignedLongLong(t.n_slots));
  for (const auto& c : cols) {
    if (!ok) break;
    if (!c.p) Py_INCREF(Py_None);
    ok = put(out, c.name, c.p ? PyLong_FromVoidPtr(const_cast<void*>(c.p)) : Py_None);
  }
  if (!ok) { Py_DECREF(out); return nullptr; }
  return Py_BuildValue("(iN)", rc, out);
}

PyObject* rank_list(const uint32_t* p, Py_ssize_t n) {                 // a copy
  npy_intp dim = n;
  PyObject* a = PyArray_SimpleNew(1, &dim, NPY_UINT32);
  if (a && n) std::memcpy(PyArray_DATA((PyArrayObject*)a), p, (size_t)n * 4);
  return a;
}
PyObject* hang_dict(const ccld_hang_verdict& v, const uint32_t* roots, Py_ssize_t cap) {
  PyObject* out = PyDict_New();
  const bool ok = out && put(out, "cls", PyLong_FromUnsignedLong(v.cls)) && put(out, "n_roots_total", PyLong_FromUnsignedLong(v.n_roots_total)) &&
                  put(out, "n_not_entered", PyLong_FromUnsignedLong(v.n_not_entered)) && put(out, "n_hung", PyLong_FromUnsignedLong(v.n_hung)) &&
                  put(out, "n_not_hung", PyLong_FromUnsignedLong(v.n_not_hung)) && put(out, "n_missing_frames", PyLong_FromUnsignedLong(v.n_missing_frames)) &&
                  put(out, "stuck_step", PyLong_FromUnsignedLong(v.stuck_step)) && put(out, "n_members", PyLong_FromUnsignedLong(v.n_members)) &&
                  put(out, "min_total", PyLong_FromUnsignedLongLong(v.min_total)) &&
                  put(out, "roots", rank_list(roots, (Py_ssize_t)v.n_roots_total < cap ? (Py_ssize_t)v.n_roots_total : cap));
  if (!ok) { Py_XDECREF(out); return nullptr; }
  return out;
}

// Room the library writes a list of up to n entries into, for one call. The lists have a largest length (members of a
// communicator, alerts of a window), so a caller's capacity beyond that needs no room.
template <class T> struct Room {
  T* const p;
  explicit Room(size_t n) : p((T*)std::malloc(n ? n * sizeof(T) : 1)) {}
  ~Room() { std::free(p); }
  Room(const Room&) = delete; Room& operator=(const Room&) = delete;
};
Py_ssize_t at_most(Py_ssize_t cap, Py_ssize_t most) { return cap < 0 ? 0 : (cap < most ? cap : most); }

// hang(context, window, communicator, op counter, roots_cap) -> (return code, dictionary)
PyObject* hang(PyObject*, PyObject* args) {
  unsigned long long h; unsigned int window, comm, seq; Py_ssize_t cap;
  if (!PyArg_ParseTuple(args, "KIIIn", &h, &window, &comm, &seq, &cap)) return nullptr;
  cap = at_most(cap, CCLD_MAX_COMM_SIZE);
  const Room<uint32_t> roots((size_t)cap);
  if (!roots.p) return PyErr_NoMemory();
  ccld_hang_verdict v;
  std::memset(&v, 0, sizeof v);
  v.roots = roots.p; v.roots_cap = (uint32_t)cap;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_hang((ccld_ctx*)h, window, comm, seq, &v);
  Py_END_ALLOW_THREADS
  if (rc != CCLD_OK) return Py_BuildValue("(iO)", rc, Py_None);
  PyObject* d = hang_dict(v, roots.p, cap);
  return d ? Py_BuildValue("(iN)", rc, d) : nullptr;
}

// hangs(context, window, cap, roots_stride) -> (return code, list of dictionaries)
PyObject* hangs(PyObject*, PyObject* args) {
  unsigned long long h; unsigned int window; Py_ssize_t cap, stride;
  if (!PyArg_ParseTuple(args, "KInn", &h, &window, &cap, &stride)) return nullptr;
  if (cap < 1) cap = 1;
  const Py_ssize_t keep = at_most(cap, CCLD_MAX_ALERTS_PER_WINDOW);
  stride = at_most(stride, CCLD_MAX_COMM_SIZE);
  const Room<ccld_hang_verdict> hv((size_t)keep);
  const Room<ccld_hang_alert> al((size_t)keep);
  const Room<uint32_t> roots((size_t)keep * (size_t)stride);
  if (!hv.p || !al.p || !roots.p) return PyErr_NoMemory();
  uint32_t n = 0;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_hangs((ccld_ctx*)h, window, al.p, hv.p, (uint32_t)keep, roots.p, (uint32_t)stride, &n);
  Py_END_ALLOW_THREADS
  if (rc != CCLD_OK) return Py_BuildValue("(iO)", rc, Py_None);
  const Py_ssize_t m = (Py_ssize_t)n < cap ? (Py_ssize_t)n : cap;
  PyObject* list = PyList_New(m);
  if (!list) return nullptr;
  for (Py_ssize_t i = 0; i < m; ++i) {
    ccld_hang_verdict v; ccld_hang_alert a;                            // alerts beyond those kept are listed as zeros
    std::memset(&v, 0, sizeof v); std::memset(&a, 0, sizeof a);
    if (i < keep) { v = hv.p[i]; a = al.p[i]; }
    PyObject* d = hang_dict(v, roots.p + (i < keep ? i * stride : 0), stride);
    if (!d || !put(d, "comm", PyLong_FromUnsignedLong(a.comm)) || !put(d, "seq", PyLong_FromUnsignedLong(a.seq)) ||
        !put(d, "age_ns", PyLong_FromLongLong(a.age_ns))) { Py_XDECREF(d); Py_DECREF(list); return nullptr; }
    PyList_SET_ITEM(list, i, d);
  }
  return Py_BuildValue("(iN)", rc, list);
}

// opset(context, window, communicator, op counter, ranks_cap) -> (return code, dictionary)
PyObject* opset(PyObject*, PyObject* args) {
  unsigned long long h; unsigned int window, comm, seq; Py_ssize_t cap;
  if (!PyArg_ParseTuple(args, "KIIIn", &h, &window, &comm, &seq, &cap)) return nullptr;
  cap = at_most(cap, CCLD_MAX_COMM_SIZE);
  const Room<uint32_t> ranks((size_t)cap);
  if (!ranks.p) return PyErr_NoMemory();
  ccld_opset_verdict v;
  std::memset(&v, 0, sizeof v);
  v.ranks = ranks.p; v.ranks_cap = (uint32_t)cap;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_opset((ccld_ctx*)h, window, comm, seq, &v);
  Py_END_ALLOW_THREADS
  if (rc != CCLD_OK) return Py_BuildValue("(iO)", rc, Py_None);
  PyObject* out = PyDict_New();
  const bool ok = out && put(out, "n_members", PyLong_FromUnsignedLong(v.n_members)) && put(out, "n_present", PyLong_FromUnsignedLong(v.n_present)) &&
                  put(out, "n_deviating_total", PyLong_FromUnsignedLong(v.n_deviating_total)) && put(out, "majority_count", PyLong_FromUnsignedLong(v.majority_count)) &&
                  put(out, "op", PyLong_FromLong(v.op)) && put(out, "algo", PyLong_FromLong(v.algo)) && put(out, "proto", PyLong_FromLong(v.proto)) &&
                  put(out, "bytes", PyLong_FromUnsignedLongLong(v.bytes)) &&
                  put(out, "ranks", rank_list(ranks.p, (Py_ssize_t)v.n_deviating_total < cap ? (Py_ssize_t)v.n_deviating_total : cap));
  if (!ok) { Py_XDECREF(out); return nullptr; }
  return Py_BuildValue("(iN)", rc, out);
}

// ranges(context, window, cap) -> (return code, dictionary of arrays)
template <class T, class F> PyObject* column_of(const ccld_comm_range* rows, Py_ssize_t n, int type, F&& field) {
  npy_intp dim = n;
  PyObject* a = PyArray_SimpleNew(1, &dim, type);
  if (a) { T* p = (T*)PyArray_DATA((PyArrayObject*)a); for (Py_ssize_t i = 0; i < n; ++i) p[i] = field(rows[i]); }
  return a;
}
PyObject* ranges(PyObject*, PyObject* args) {
  unsigned long long h; unsigned int window; Py_ssize_t cap;
  if (!PyArg_ParseTuple(args, "KIn", &h, &window, &cap)) return nullptr;
  cap = at_most(cap, (Py_ssize_t)0xFFFFFFFFu);
  const Room<ccld_comm_range> room((size_t)cap);
  if (!room.p) return PyErr_NoMemory();
  ccld_comm_range* const rows = room.p;
  uint32_t total = 0;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_ranges((ccld_ctx*)h, window, rows, (uint32_t)cap, &total);
  Py_END_ALLOW_THREADS
  if (rc != CCLD_OK) return Py_BuildValue("(iO)", rc, Py_None);
  const Py_ssize_t n = (Py_ssize_t)total < cap ? (Py_ssize_t)total : cap;
  PyObject* out = PyDict_New();
  typedef const ccld_comm_range& Row;
  const bool ok = out && put(out, "comm", column_of<uint32_t>(rows, n, NPY_UINT32, [](Row r) { return r.comm; })) &&
                  put(out, "n", column_of<uint32_t>(rows, n, NPY_UINT32, [](Row r) { return r.n; })) &&
                  put(out, "seq_lo", column_of<uint32_t>(rows, n, NPY_UINT32, [](Row r) { return r.seq_lo; })) &&
                  put(out, "n_seq", column_of<uint32_t>(rows, n, NPY_UINT32, [](Row r) { return r.n_seq; })) &&
                  put(out, "group0", column_of<uint64_t>(rows, n, NPY_UINT64, [](Row r) { return r.group0; })) &&
                  put(out, "slot0", column_of<uint64_t>(rows, n, NPY_UINT64, [](Row r) { return r.slot0; }));
  if (!ok) { Py_XDECREF(out); return nullptr; }
  return Py_BuildValue("(iN)", rc, out);
}

// rates(context, records, rank, t_enter, t_exit, ranks, ticks, tick_off, tick_ns, send_count, recv_count, send_chg, recv_chg):
// device addresses -> return code
PyObject* rates(PyObject*, PyObject* const* args, Py_ssize_t n) {
  unsigned long long a[13];
  if (n != 13) { PyErr_SetString(PyExc_TypeError, "rates takes 13 whole numbers"); return nullptr; }
  for (int i = 0; i < 13; ++i) {
    a[i] = PyLong_AsUnsignedLongLongMask(args[i]);
    if (a[i] == (unsigned long long)-1 && PyErr_Occurred()) return nullptr;
  }
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_rates((ccld_ctx*)a[0], a[1], (const uint32_t*)a[2], (const int64_t*)a[3], (const int64_t*)a[4], (uint32_t)a[5], a[6], (const uint64_t*)a[7],
               (const int64_t*)a[8], (const uint32_t*)a[9], (const uint32_t*)a[10], (uint32_t*)a[11], (uint32_t*)a[12]);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

PyMethodDef methods[] = {{"setup", setup, METH_VARARGS, "Addresses of the library's functions, names of fields."},
                         {"verdict", verdict, METH_VARARGS, "ccld_get_verdict_columns as a dictionary of arrays."},
                         {"upload", upload, METH_VARARGS, "ccld_trace_upload of numpy columns."},
                         {"rank_stats", rank_stats, METH_VARARGS, "ccld_take_rank_stats as a dictionary of arrays."},
                         {"optable", optable, METH_VARARGS, "ccld_take_optable as a dictionary of arrays."},
                         {"table", table, METH_VARARGS, "ccld_get_optable as a dictionary of device addresses."},
                         {"hang", hang, METH_VARARGS, "ccld_locate_hang as a dictionary."},
                         {"hangs", hangs, METH_VARARGS, "ccld_locate_hangs as a list of dictionaries."},
                         {"opset", opset, METH_VARARGS, "ccld_opset_check as a dictionary."},
                         {"ranges", ranges, METH_VARARGS, "ccld_get_ranges as a dictionary of arrays."},
                         {"rates", (PyCFunction)(void (*)(void))rates, METH_FASTCALL, "ccld_derive_rates on device addresses."},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__binding(void) {
  import_array();
  return PyModule_Create(&module);
}
