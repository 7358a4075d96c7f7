/* The hot entry points of libfastav.so for Python: tensors in, status out.  Argument marshalling only.
 *
 * A prune call takes about twenty pointers.  Through ctypes that is 6.5 us a call, more than a small call's kernels take to
 * launch; a tensor's data_ptr() called from C is 60 ns.  The library itself stays free of Python: the functions come in
 * as addresses of the ctypes handle that loaded it.  As through ctypes, other threads run during a call: a launch waits while
 * the stream's queue is full, and what empties the queue may be a Python callback. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <stdint.h>

#include "fastav.h"

static PyObject* s_data_ptr;
static PyObject* s_nbytes;

/* An address given as an int (0 on error, with the exception set). */
static void* address(PyObject* o) { return PyLong_AsVoidPtr(o); }

/* Device pointer of a tensor; None is NULL. */
static int pointer(PyObject* o, void** out) {
  if (o == Py_None) {
    *out = NULL;
    return 0;
  }
  PyObject* r = PyObject_VectorcallMethod(s_data_ptr, &o, 1 | PY_VECTORCALL_ARGUMENTS_OFFSET, NULL);
  if (!r) return -1;
  *out = PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

static int pointers(PyObject* const* a, int n, void** out) {
  for (int i = 0; i < n; ++i)
    if (pointer(a[i], &out[i]) != 0) return -1;
  return 0;
}

static int size_of(PyObject* o, size_t* out) {
  *out = 0;
  if (o == Py_None) return 0;
  PyObject* r = PyObject_GetAttr(o, s_nbytes);
  if (!r) return -1;
  *out = PyLong_AsSize_t(r);
  Py_DECREF(r);
  return *out == (size_t)-1 && PyErr_Occurred() ? -1 : 0;
}

static int expect(const char* name, Py_ssize_t got, Py_ssize_t want) {
  if (got == want) return 0;
  PyErr_Format(PyExc_TypeError, "%s takes %zd arguments, got %zd", name, want, got);
  return -1;
}

/* (function, params, 18 tensors in the order of fastav_prune, workspace, device_status, stream) */
static PyObject* prune(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void *f, *p, *t[18], *ws, *status, *stream;
  size_t bytes;
  if (expect("prune", n, 23) || ((f = address(a[0])) == NULL) || ((p = address(a[1])) == NULL) || pointers(a + 2, 18, t) ||
      pointer(a[20], &ws) || size_of(a[20], &bytes) || pointer(a[21], &status))
    return NULL;
  stream = address(a[22]);
  if (PyErr_Occurred()) return NULL;
  int32_t rc;
  Py_BEGIN_ALLOW_THREADS
  rc = ((__typeof__(&fastav_prune))f)(p, t[0], t[1], t[2], t[3], t[4], t[5], t[6], t[7], t[8], t[9], t[10], t[11], t[12], t[13], t[14], t[15],
                                      t[16], t[17], ws, bytes, status, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

/* (function, params, keep_mask, cu_seqlens, keep_idx_out, cu_keep_out, workspace, device_status, stream) */
static PyObject* select_mask(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void *f, *p, *t[4], *ws, *status, *stream;
  size_t bytes;
  if (expect("select_mask", n, 9) || ((f = address(a[0])) == NULL) || ((p = address(a[1])) == NULL) || pointers(a + 2, 4, t) ||
      pointer(a[6], &ws) || size_of(a[6], &bytes) || pointer(a[7], &status))
    return NULL;
  stream = address(a[8]);
  if (PyErr_Occurred()) return NULL;
  int32_t rc;
  Py_BEGIN_ALLOW_THREADS
  rc = ((__typeof__(&fastav_select_mask))f)(p, t[0], t[1], t[2], t[3], ws, bytes, status, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

/* (function, params, keep_idx, cu_keep, cu_seqlens, hidden in/out, pos in/out, k in/out, v in/out, device_status, stream) */
static PyObject* compact(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void *f, *p, *t[12], *stream;
  if (expect("compact", n, 15) || ((f = address(a[0])) == NULL) || ((p = address(a[1])) == NULL) || pointers(a + 2, 12, t)) return NULL;
  stream = address(a[14]);
  if (PyErr_Occurred()) return NULL;
  int32_t rc;
  Py_BEGIN_ALLOW_THREADS
  rc = ((__typeof__(&fastav_compact))f)(p, t[0], t[1], t[2], t[3], t[4], t[5], t[6], t[7], t[8], t[9], t[10], t[11], stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {
    {"prune", (PyCFunction)(void (*)(void))prune, METH_FASTCALL, "fastav_prune"},
    {"select_mask", (PyCFunction)(void (*)(void))select_mask, METH_FASTCALL, "fastav_select_mask"},
    {"compact", (PyCFunction)(void (*)(void))compact, METH_FASTCALL, "fastav_compact"},
    {NULL, NULL, 0, NULL},
};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", "Argument marshalling for libfastav.so.", -1, methods};

PyMODINIT_FUNC PyInit__binding(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_nbytes = PyUnicode_InternFromString("nbytes");
  return s_data_ptr && s_nbytes ? PyModule_Create(&module) : NULL;
}
