/*
 * The per-step calls of the binding without ctypes: mix_apply, mix_set_slot_map, mix_set_request_map.
 *
 * An eager decode step is two of these calls and two kernels, and the host sets its pace: of 4.2 us for an apply, 2.2 were
 * the launch, the rest attribute look-ups in Python and ctypes' conversions.  The checks are the binding's own, made here on
 * the same tensor attributes; a call that fails one raises what the Python code raised.  The GIL is released round the call
 * into the library, as ctypes releases it: a launch can wait for room in a full queue, and a copy from pageable memory for
 * everything in front of it, which may be a host function that itself needs the GIL.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "mix.h"

static PyObject *s_is_cuda, *s_dtype, *s_is_contiguous, *s_data_ptr, *s_size, *s_numel, *zero;   /* interned names */
static PyObject *t_bf16, *t_int32;                                                           /* torch dtypes */
static PyObject *get_device, *get_stream;                                                                /* torch._C functions */

static int flag(PyObject* t, PyObject* name, int call) {        /* truth of an attribute or of a method's answer; -1: error set */
  PyObject* v = call ? PyObject_CallMethodNoArgs(t, name) : PyObject_GetAttr(t, name);
  if (!v) return -1;
  const int r = PyObject_IsTrue(v);
  Py_DECREF(v);
  return r;
}
static int has_dtype(PyObject* t, PyObject* dtype) {
  PyObject* v = PyObject_GetAttr(t, s_dtype);
  if (!v) return -1;
  Py_DECREF(v);                                                 /* (dtypes live as long as torch) */
  return v == dtype;
}
static int number(PyObject* v, long long* out) {                /* steals v; -1: error set */
  if (!v) return -1;
  *out = PyLong_AsLongLong(v);
  Py_DECREF(v);
  return *out == -1 && PyErr_Occurred() ? -1 : 0;
}
static int data_ptr(PyObject* t, void** out) {
  PyObject* v = PyObject_CallMethodNoArgs(t, s_data_ptr);
  if (!v) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !*out && PyErr_Occurred() ? -1 : 0;
}
/* None: torch's current stream; a torch stream (cuda_stream) or a raw handle otherwise */
static int stream_of(PyObject* s, void** out) {
  PyObject* v;
  if (s == Py_None) {
    PyObject* dev = PyObject_CallNoArgs(get_device);
    if (!dev) return -1;
    v = PyObject_CallOneArg(get_stream, dev);
    Py_DECREF(dev);
  } else {
    v = PyObject_GetAttrString(s, "cuda_stream");
    if (!v) {
      PyErr_Clear();
      v = PyNumber_Long(s);
    }
  }
  if (!v) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !*out && PyErr_Occurred() ? -1 : 0;
}
static int context(PyObject* o, mix_ctx** out) {
  *out = (mix_ctx*)PyLong_AsVoidPtr(o);
  return !*out && PyErr_Occurred() ? -1 : 0;
}

/* apply(ctx, hidden, scores_out | None, T | None, stream | None) -> status */
static PyObject* fast_apply(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  mix_ctx* c;
  void *h, *scores = NULL, *stream;
  long long T;
  if (n != 5) return PyErr_Format(PyExc_TypeError, "apply takes 5 arguments");
  if (context(a[0], &c) < 0) return NULL;
  const int ok1 = has_dtype(a[1], t_bf16), ok2 = ok1 > 0 ? flag(a[1], s_is_cuda, 0) : ok1, ok3 = ok2 > 0 ? flag(a[1], s_is_contiguous, 1) : ok2;
  if (ok3 < 0) return NULL;
  if (!ok3) return PyErr_Format(PyExc_AssertionError, "hidden must be a contiguous CUDA bfloat16 tensor");
  if (data_ptr(a[1], &h) < 0) return NULL;
  if (a[3] == Py_None) {
    if (number(PyObject_CallMethodOneArg(a[1], s_size, zero), &T) < 0) return NULL;
  } else if (number(PyNumber_Long(a[3]), &T) < 0) {
    return NULL;
  }
  if (a[2] != Py_None) {
    const int k1 = flag(a[2], s_is_cuda, 0), k2 = k1 > 0 ? flag(a[2], s_is_contiguous, 1) : k1;
    if (k2 < 0) return NULL;
    if (!k2) return PyErr_Format(PyExc_ValueError, "expected a contiguous CUDA tensor");
    if (data_ptr(a[2], &scores) < 0) return NULL;
  }
  if (stream_of(a[4], &stream) < 0) return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = mix_apply(c, h, (int)T, (float*)scores, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

/* set_slot_map(ctx, token_slot int32 tensor, T_live | None, stream | None) -> status */
static PyObject* fast_set_slot_map(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  mix_ctx* c;
  void *src, *stream;
  long long T;
  if (n != 4) return PyErr_Format(PyExc_TypeError, "set_slot_map takes 4 arguments");
  if (context(a[0], &c) < 0) return NULL;
  const int ok1 = has_dtype(a[1], t_int32), ok2 = ok1 > 0 ? flag(a[1], s_is_contiguous, 1) : ok1;
  if (ok2 < 0) return NULL;
  if (!ok2) return PyErr_Format(PyExc_AssertionError, "token_slot must be a contiguous int32 tensor");
  const int cuda = flag(a[1], s_is_cuda, 0);
  if (cuda < 0 || data_ptr(a[1], &src) < 0) return NULL;
  if (number(a[2] == Py_None ? PyObject_CallMethodNoArgs(a[1], s_numel) : PyNumber_Index(a[2]), &T) < 0) return NULL;
  if (stream_of(a[3], &stream) < 0) return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = mix_set_slot_map(c, (const int*)src, (int)T, cuda, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

/* set_request_map(ctx, token_req, req_slot, T_live | None, stream | None) -> status */
static PyObject* fast_set_request_map(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  mix_ctx* c;
  void *req, *slots, *stream;
  long long T, n_req;
  if (n != 5) return PyErr_Format(PyExc_TypeError, "set_request_map takes 5 arguments");
  if (context(a[0], &c) < 0) return NULL;
  const int cuda = flag(a[1], s_is_cuda, 0);
  if (cuda < 0 || data_ptr(a[1], &req) < 0 || data_ptr(a[2], &slots) < 0) return NULL;
  if (number(a[3] == Py_None ? PyObject_CallMethodNoArgs(a[1], s_numel) : PyNumber_Index(a[3]), &T) < 0) return NULL;
  if (number(PyObject_CallMethodNoArgs(a[2], s_numel), &n_req) < 0) return NULL;
  if (stream_of(a[4], &stream) < 0) return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = mix_set_request_map(c, (const int*)req, (int)T, (const int*)slots, (int)n_req, cuda, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {
    {"apply", (PyCFunction)(void (*)(void))fast_apply, METH_FASTCALL, NULL},
    {"set_slot_map", (PyCFunction)(void (*)(void))fast_set_slot_map, METH_FASTCALL, NULL},
    {"set_request_map", (PyCFunction)(void (*)(void))fast_set_request_map, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__fastcall(void) {
  PyObject* torch = PyImport_ImportModule("torch");
  if (!torch) return NULL;
  PyObject* tc = PyObject_GetAttrString(torch, "_C");
  s_is_cuda = PyUnicode_InternFromString("is_cuda");
  s_dtype = PyUnicode_InternFromString("dtype");
  s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_size = PyUnicode_InternFromString("size");
  s_numel = PyUnicode_InternFromString("numel");
  zero = PyLong_FromLong(0);
  t_bf16 = PyObject_GetAttrString(torch, "bfloat16");
  t_int32 = PyObject_GetAttrString(torch, "int32");
  if (tc) {
    get_device = PyObject_GetAttrString(tc, "_cuda_getDevice");
    get_stream = PyObject_GetAttrString(tc, "_cuda_getCurrentRawStream");
  }
  if (!tc || !t_bf16 || !t_int32 || !get_device || !get_stream) return NULL;
  return PyModule_Create(&module);
}
