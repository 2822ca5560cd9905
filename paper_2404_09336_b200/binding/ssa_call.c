/* Python calls -> C entry points of libssa: addresses, strides and sizes are read off the argument objects here instead of
 * in Python and ctypes, which took longer than the kernels of a small call (decode_attn_sparse up to the entry point: 9.4 us,
 * 2.3 us with this; whole calls on a B200: 11.2 -> 4.6 us for 2 requests of 201 rows, decode_step of one short request 7.9
 * -> 3.5 us, refs_to_index and decode_attn_sparse 24.4 -> 13.8 us, the kernels' own time).
 *
 * bind(addresses) takes the entry points of one loaded library, so that another can be loaded next to it, and the classes
 * of the descriptor structures.  The calls take what the wrappers in ssa.py document: tensors (anything with data_ptr()) or
 * None, integers, descriptor structures, and the stream as an integer; they return the status code.  The GIL is released
 * while an entry point runs, as it was by ctypes. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "ssa.h"

#define ENTRY_POINTS(X)                                                                                              \
  X(spans_to_index) X(decode_attn_sparse) X(decode_attn_spans) X(decode_attn_sparse_multiq) X(decode_attn_dense_multiq) \
  X(spans_to_blockmask) X(decode_attn_blockmask) X(decode_attn_sparse_paged) X(decode_attn_dense_paged)               \
  X(refs_to_index) X(refs_to_spans) X(decode_step) X(decode_attn_sparse_noalloc) X(decode_attn_dense)

/* Structures that a caller fills.  Only instances of the class that bind() was given for one are taken (without a class:
 * buffers of its exact size), so that no other structure and no other buffer is read as sizes and strides. */
enum { kDesc, kStep, kPaging, kStructures };
static const char* const structure_name[kStructures] = {"ssa_attn_desc", "ssa_step", "ssa_paging"};
static const size_t structure_size[kStructures] = {sizeof(ssa_attn_desc), sizeof(ssa_step), sizeof(ssa_paging)};

typedef struct {
#define X(name) __typeof__(&ssa_##name) name;
  ENTRY_POINTS(X)
#undef X
  PyObject* structure[kStructures];   /* classes; NULL: bind() was given none */
  PyObject *s_data_ptr, *s_numel, *s_element_size, *s_stride, *s_shape, *s_zero;
} State;

/* ---- arguments ---- */
enum { kMost = 24 };
typedef struct {
  void* p[kMost];          /* addresses in the order of the format's D, t, r and w */
  int64_t v[kMost];        /* integers in the order of its i, n, r (row stride) and w (bytes) */
  Py_buffer held[4];
  int n_held;
} Args;

static int integer(PyObject* o, int64_t* out) {
  if (PyLong_Check(o)) {
    *out = (int64_t)PyLong_AsUnsignedLongLongMask(o);
  } else {
    PyObject* n = PyNumber_Long(o);
    if (!n) return -1;
    *out = (int64_t)PyLong_AsUnsignedLongLongMask(n);
    Py_DECREF(n);
  }
  return PyErr_Occurred() ? -1 : 0;
}

static int integer_of(PyObject* o, PyObject* method, PyObject* arg, int64_t* out) {
  PyObject* r = arg ? PyObject_CallMethodOneArg(o, method, arg) : PyObject_CallMethodNoArgs(o, method);
  if (!r) return -1;
  const int rc = integer(r, out);
  Py_DECREF(r);
  return rc;
}

static int address(const State* st, PyObject* o, void** out) {
  int64_t at = 0;
  if (o != Py_None && integer_of(o, st->s_data_ptr, NULL, &at) < 0) return -1;
  *out = (void*)(uintptr_t)at;
  return 0;
}

/* shape[0] and the elements between consecutive rows (a one-row tensor may carry any stride for that dimension) */
static int rows_of(const State* st, PyObject* o, int64_t* rows, int64_t* stride) {
  PyObject* shape = PyObject_GetAttr(o, st->s_shape);
  if (!shape) return -1;
  int rc = -1;
  PyObject* first = PySequence_GetItem(shape, 0);
  if (first && integer(first, rows) == 0) {
    if (*rows > 1) {
      rc = integer_of(o, st->s_stride, st->s_zero, stride);
    } else {
      PyObject* second = PySequence_GetItem(shape, 1);
      if (second) { rc = integer(second, stride); Py_DECREF(second); }
    }
  }
  Py_XDECREF(first);
  Py_DECREF(shape);
  return rc;
}

static void release(Args* x) {
  for (int i = 0; i < x->n_held; ++i) PyBuffer_Release(&x->held[i]);
}

static int structure(const State* st, int which, PyObject* o, Py_buffer* held) {
  const int is = st->structure[which] ? PyObject_IsInstance(o, st->structure[which]) : 1;
  if (is < 0) return -1;
  if (is && PyObject_GetBuffer(o, held, PyBUF_SIMPLE) < 0) return -1;
  if (is && (st->structure[which] ? (size_t)held->len >= structure_size[which] : (size_t)held->len == structure_size[which])) return 0;
  if (is) PyBuffer_Release(held);
  PyErr_Format(PyExc_TypeError, "%s wanted, not %.80s", structure_name[which], Py_TYPE(o)->tp_name);
  return -1;
}

/* format: D ssa_attn_desc, S ssa_step, P ssa_paging or None, t tensor or None, r tensor or None and its row stride,
 * w tensor or None and its bytes, i integer, n tensor and its number of elements. */
static int parse(const State* st, Args* x, const char* name, const char* format, PyObject* const* a, Py_ssize_t n) {
  int np = 0, nv = 0;
  x->n_held = 0;
  if (n != (Py_ssize_t)strlen(format)) {
    PyErr_Format(PyExc_TypeError, "%s: %zd arguments, %zd wanted", name, n, (Py_ssize_t)strlen(format));
    return -1;
  }
  for (Py_ssize_t i = 0; i < n; ++i) {
    PyObject* o = a[i];
    int64_t bytes = 0;
    switch (format[i]) {
      case 'P':
        if (o == Py_None) { x->p[np++] = NULL; break; }  /* fall through */
      case 'D':
      case 'S':
        if (structure(st, format[i] == 'D' ? kDesc : format[i] == 'S' ? kStep : kPaging, o, &x->held[x->n_held]) < 0) goto bad;
        x->p[np++] = x->held[x->n_held++].buf;
        break;
      case 't':
        if (address(st, o, &x->p[np++]) < 0) goto bad;
        break;
      case 'n':
        if (address(st, o, &x->p[np++]) < 0 || integer_of(o, st->s_numel, NULL, &x->v[nv++]) < 0) goto bad;
        break;
      case 'r':
        if (address(st, o, &x->p[np++]) < 0) goto bad;
        x->v[nv] = 0;
        if (o != Py_None && rows_of(st, o, &bytes, &x->v[nv]) < 0) goto bad;
        ++nv;
        break;
      case 'w':
        if (address(st, o, &x->p[np++]) < 0) goto bad;
        x->v[nv] = 0;
        if (o != Py_None) {
          if (integer_of(o, st->s_numel, NULL, &x->v[nv]) < 0 || integer_of(o, st->s_element_size, NULL, &bytes) < 0) goto bad;
          x->v[nv] *= bytes;
        }
        ++nv;
        break;
      default:
        if (integer(o, &x->v[nv++]) < 0) goto bad;
    }
  }
  return 0;
bad:
  release(x);
  return -1;
}

#define CALL(name, format, expression)                                                               \
  static PyObject* call_##name(PyObject* self, PyObject* const* a, Py_ssize_t n) {                   \
    const State* st = (const State*)PyModule_GetState(self);                                         \
    Args x;                                                                                          \
    int32_t rc;                                                                                      \
    if (!st->name) { PyErr_SetString(PyExc_RuntimeError, "no library bound"); return NULL; }         \
    if (parse(st, &x, #name, format, a, n) < 0) return NULL;                                   \
    void** const p = x.p;                                                                            \
    const int64_t* const v = x.v;                                                                    \
    (void)v;                                                                                         \
    Py_BEGIN_ALLOW_THREADS                                                                           \
    rc = st->name expression;                                                                        \
    Py_END_ALLOW_THREADS                                                                             \
    release(&x);                                                                                     \
    return PyLong_FromLong(rc);                                                                      \
  }
#define I(k) ((int32_t)v[k])
#define STREAM(k) ((void*)(uintptr_t)v[k])

/* the order of the arguments is that of the entry points; the stream comes last */
CALL(spans_to_index, "ttnrtti", (p[0], p[1], p[2], I(0), p[3], I(1), p[4], p[5], STREAM(2)))
CALL(decode_attn_sparse, "Dtttt" "rtitt" "wti",
     (p[0], p[1], p[2], p[3], p[4], p[5], I(0), p[6], I(1), p[7], p[8], p[9], (size_t)v[2], p[10], STREAM(3)))
CALL(decode_attn_spans, "Dtttt" "ttii" "ttrt" "wti",
     (p[0], p[1], p[2], p[3], p[4], p[5], p[6], I(0), I(1), p[7], p[8], p[9], I(2), p[10], p[11], (size_t)v[3], p[12], STREAM(4)))
CALL(decode_attn_sparse_multiq, "Diii" "tttt" "rtitt" "wti",
     (p[0], I(0), v[1], v[2], p[1], p[2], p[3], p[4], p[5], I(3), p[6], I(4), p[7], p[8], p[9], (size_t)v[5], p[10], STREAM(6)))
CALL(decode_attn_dense_multiq, "Diii" "tttt" "tt" "wti",
     (p[0], I(0), v[1], v[2], p[1], p[2], p[3], p[4], p[5], p[6], p[7], (size_t)v[3], p[8], STREAM(4)))
CALL(spans_to_blockmask, "ttni" "rttti",
     (p[0], p[1], p[2], I(0), I(1), p[3], p[4], I(2), p[5], p[6], STREAM(3)))
CALL(decode_attn_blockmask, "Dtttt" "rttii" "tt" "wti",
     (p[0], p[1], p[2], p[3], p[4], p[5], p[6], I(0), p[7], I(1), I(2), p[8], p[9], p[10], (size_t)v[3], p[11], STREAM(4)))
CALL(decode_attn_sparse_paged, "DtttPt" "rtitt" "wti",
     (p[0], p[1], p[2], p[3], p[4], p[5], p[6], I(0), p[7], I(1), p[8], p[9], p[10], (size_t)v[2], p[11], STREAM(3)))
CALL(decode_attn_dense_paged, "DtttPt" "tt" "wti",
     (p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], p[8], (size_t)v[0], p[9], STREAM(1)))
CALL(decode_step, "DSi", (p[0], p[1], STREAM(0)))
CALL(decode_attn_sparse_noalloc, "Dtttt" "rtitt" "ti",
     (p[0], p[1], p[2], p[3], p[4], p[5], I(0), p[6], I(1), p[7], p[8], p[9], STREAM(2)))
CALL(decode_attn_dense, "Dtttt" "tt" "wti",
     (p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], (size_t)v[0], p[8], STREAM(1)))

static ssa_anchor_tables tables(void* const* p) {
  ssa_anchor_tables t;
  memset(&t, 0, sizeof t);
  t.line_offsets = p[0]; t.lines = p[1]; t.anchor_offsets = p[2]; t.anchor_line = p[3]; t.ref_offsets = p[4];
  t.refs = p[5]; t.prefix_len = p[6]; t.line_start = p[7]; t.ctx_lens = p[8];
  return t;
}
CALL(refs_to_index, "ttttttttn" "rtti",
     (&(const ssa_anchor_tables[]){tables(p)}[0], I(0), p[9], I(1), p[10], p[11], STREAM(2)))
CALL(refs_to_spans, "ttttttttn" "ttiti",
     (&(const ssa_anchor_tables[]){tables(p)}[0], I(0), p[9], p[10], I(1), p[11], STREAM(2)))

static PyObject* bind_library(PyObject* self, PyObject* addresses) {
  State* st = (State*)PyModule_GetState(self);
#define X(name)                                                                     \
  {                                                                                 \
    PyObject* o = PyMapping_GetItemString(addresses, "ssa_" #name);                 \
    int64_t at = 0;                                                                 \
    if (!o) return NULL;                                                            \
    const int rc = integer(o, &at);                                                 \
    Py_DECREF(o);                                                                   \
    if (rc < 0) return NULL;                                                        \
    st->name = (__typeof__(st->name))(uintptr_t)at;                                 \
  }
  ENTRY_POINTS(X)
#undef X
  for (int i = 0; i < kStructures; ++i) {
    PyObject* type = PyMapping_GetItemString(addresses, structure_name[i]);
    if (!type) {
      if (!PyErr_ExceptionMatches(PyExc_KeyError)) return NULL;
      PyErr_Clear();
    }
    Py_XSETREF(st->structure[i], type);
  }
  Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"bind", bind_library, METH_O, "bind(addresses): the entry points to call and the classes of their structures, by name"},
#define X(name) {#name, (PyCFunction)(void (*)(void))call_##name, METH_FASTCALL, "ssa_" #name},
    ENTRY_POINTS(X)
#undef X
    {NULL, NULL, 0, NULL}};

static int start(PyObject* m) {
  State* st = (State*)PyModule_GetState(m);
  return (st->s_data_ptr = PyUnicode_InternFromString("data_ptr")) && (st->s_numel = PyUnicode_InternFromString("numel")) &&
                 (st->s_element_size = PyUnicode_InternFromString("element_size")) &&
                 (st->s_stride = PyUnicode_InternFromString("stride")) && (st->s_shape = PyUnicode_InternFromString("shape")) &&
                 (st->s_zero = PyLong_FromLong(0))
             ? 0
             : -1;
}

static PyModuleDef_Slot slots[] = {{Py_mod_exec, start}, {0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_ssa_call", "Calls into libssa", sizeof(State), methods, slots,
                                    NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__ssa_call(void) { return PyModuleDef_Init(&module); }
