/* Argument marshalling of the per-layer entry points for Python: a CPython module that turns the binding's arguments into one
 * C call.  Bound by interpreter overhead: through ctypes the smallest decode call spent 7.3 us on the host, 1.6 of them on the
 * conversion of its nineteen arguments and 1.4 on the pointers of its nine tensors; the launch itself takes 2.9.  Here 5.1 us,
 * below what the GPU takes (6.5); an append 5.5 -> 4.0.  The other entry points are called rarely and stay with ctypes.
 * The entry points' addresses come from the ctypes library (bind), so there is one copy of the library in the process. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "../../include/q4kv.h"

static int (*f_append)(const q4kv_spec*, void*, int32_t, int32_t, const q4kv_batch*, const int32_t*, const int32_t*, int32_t,
                       const void*, const void*, int32_t*, void*);
static int (*f_decode)(const q4kv_spec*, const void*, int32_t, int32_t, const q4kv_batch*, const int32_t*, int32_t, int32_t,
                       const void*, float, void*, int32_t, float*, void*, size_t, int32_t*, void*);
static int (*f_append_decode)(const q4kv_spec*, void*, int32_t, int32_t, const q4kv_batch*, const int32_t*, int32_t, int32_t,
                              const void*, const void*, const void*, float, void*, int32_t, float*, void*, size_t, int32_t*,
                              void*);
static int (*f_prefill)(const q4kv_spec*, const void*, int32_t, int32_t, const q4kv_batch*, const int32_t*, const int32_t*,
                        int32_t, int32_t, int32_t, int32_t, const void*, float, void*, int32_t, float*, void*, size_t, int32_t*,
                        void*);
static PyObject *s_is_cuda, *s_is_contiguous, *s_data_ptr, *s_nbytes;

/* A device pointer: None, an integer, or a contiguous CUDA tensor. */
static int get_ptr(PyObject* o, void** out) {
  if (o == Py_None) { *out = NULL; return 1; }
  if (PyLong_Check(o)) { *out = PyLong_AsVoidPtr(o); return !(*out == NULL && PyErr_Occurred()); }
  PyObject* r = PyObject_GetAttr(o, s_is_cuda);
  if (!r) return 0;
  int ok = PyObject_IsTrue(r);
  Py_DECREF(r);
  if (ok > 0) {
    if (!(r = PyObject_CallMethodNoArgs(o, s_is_contiguous))) return 0;
    ok = PyObject_IsTrue(r);
    Py_DECREF(r);
  }
  if (ok < 0) return 0;
  if (!ok) { PyErr_SetString(PyExc_AssertionError, "device pointers come from contiguous CUDA tensors"); return 0; }
  if (!(r = PyObject_CallMethodNoArgs(o, s_data_ptr))) return 0;
  *out = PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return !(*out == NULL && PyErr_Occurred());
}
static int get_i32(PyObject* o, int32_t* out) {
  const unsigned long v = PyLong_AsUnsignedLongMask(o);
  *out = (int32_t)(uint32_t)v;
  return !(v == (unsigned long)-1 && PyErr_Occurred());
}
static int get_f32(PyObject* o, float* out) {
  const double v = PyFloat_AsDouble(o);
  *out = (float)v;
  return !(v == -1.0 && PyErr_Occurred());
}
static int get_bytes(PyObject* o, size_t* out) {           /* of a tensor */
  PyObject* r = PyObject_GetAttr(o, s_nbytes);
  if (!r) return 0;
  *out = PyLong_AsSize_t(r);
  Py_DECREF(r);
  return !(*out == (size_t)-1 && PyErr_Occurred());
}
/* The bytes of a ctypes structure, copied. */
static int get_struct(PyObject* o, void* out, size_t size) {
  Py_buffer v;
  if (PyObject_GetBuffer(o, &v, PyBUF_SIMPLE) != 0) return 0;
  const int ok = (size_t)v.len == size;
  if (ok) memcpy(out, v.buf, size);
  PyBuffer_Release(&v);
  if (!ok) PyErr_SetString(PyExc_TypeError, "a Spec and a Batch are expected");
  return ok;
}
static int count(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return 1;
  PyErr_Format(PyExc_TypeError, "%zd arguments expected, %zd given", want, n);
  return 0;
}

/* spec, pool, n_blocks, layer, batch: the first five arguments of all four */
typedef struct { q4kv_spec spec; q4kv_batch batch; void* pool; int32_t n_blocks, layer; } Head;
static int get_head(PyObject* const* a, Head* h) {
  return get_struct(a[0], &h->spec, sizeof h->spec) && get_ptr(a[1], &h->pool) && get_i32(a[2], &h->n_blocks) &&
         get_i32(a[3], &h->layer) && get_struct(a[4], &h->batch, sizeof h->batch);
}
/* q, softmax_scale, out, out_dtype, lse, workspace, status_flags, stream: the last eight of the attention calls */
typedef struct { void *q, *out, *lse, *ws, *flags, *stream; float scale; int32_t out_dtype; size_t ws_bytes; } Tail;
static int get_tail(PyObject* const* a, Tail* t) {
  return get_ptr(a[0], &t->q) && get_f32(a[1], &t->scale) && get_ptr(a[2], &t->out) && get_i32(a[3], &t->out_dtype) &&
         get_ptr(a[4], &t->lse) && get_ptr(a[5], &t->ws) && get_bytes(a[5], &t->ws_bytes) && get_ptr(a[6], &t->flags) &&
         get_ptr(a[7], &t->stream);
}

static PyObject* append(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Head h;
  void *pos, *offs, *k, *v, *flags, *stream;
  int32_t total;
  int rc;
  if (!count(n, 12) || !get_head(a, &h) || !get_ptr(a[5], &pos) || !get_ptr(a[6], &offs) || !get_i32(a[7], &total) ||
      !get_ptr(a[8], &k) || !get_ptr(a[9], &v) || !get_ptr(a[10], &flags) || !get_ptr(a[11], &stream))
    return NULL;
  Py_BEGIN_ALLOW_THREADS
  rc = f_append(&h.spec, h.pool, h.n_blocks, h.layer, &h.batch, pos, offs, total, k, v, flags, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}
static PyObject* decode(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Head h;
  Tail t;
  void* lens;
  int32_t max_kv, window;
  int rc;
  if (!count(n, 16) || !get_head(a, &h) || !get_ptr(a[5], &lens) || !get_i32(a[6], &max_kv) || !get_i32(a[7], &window) ||
      !get_tail(a + 8, &t))
    return NULL;
  Py_BEGIN_ALLOW_THREADS
  rc = f_decode(&h.spec, h.pool, h.n_blocks, h.layer, &h.batch, lens, max_kv, window, t.q, t.scale, t.out, t.out_dtype, t.lse,
                t.ws, t.ws_bytes, t.flags, t.stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}
static PyObject* append_decode(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Head h;
  Tail t;
  void *lens, *k, *v;
  int32_t max_kv, window;
  int rc;
  if (!count(n, 18) || !get_head(a, &h) || !get_ptr(a[5], &lens) || !get_i32(a[6], &max_kv) || !get_i32(a[7], &window) ||
      !get_ptr(a[8], &k) || !get_ptr(a[9], &v) || !get_tail(a + 10, &t))
    return NULL;
  Py_BEGIN_ALLOW_THREADS
  rc = f_append_decode(&h.spec, h.pool, h.n_blocks, h.layer, &h.batch, lens, max_kv, window, k, v, t.q, t.scale, t.out,
                       t.out_dtype, t.lse, t.ws, t.ws_bytes, t.flags, t.stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}
static PyObject* prefill(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Head h;
  Tail t;
  void *lens, *offs;
  int32_t total, max_q, max_kv, window;
  int rc;
  if (!count(n, 19) || !get_head(a, &h) || !get_ptr(a[5], &lens) || !get_ptr(a[6], &offs) || !get_i32(a[7], &total) ||
      !get_i32(a[8], &max_q) || !get_i32(a[9], &max_kv) || !get_i32(a[10], &window) || !get_tail(a + 11, &t))
    return NULL;
  Py_BEGIN_ALLOW_THREADS
  rc = f_prefill(&h.spec, h.pool, h.n_blocks, h.layer, &h.batch, lens, offs, total, max_q, max_kv, window, t.q, t.scale, t.out,
                 t.out_dtype, t.lse, t.ws, t.ws_bytes, t.flags, t.stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}
/* bind(append, decode, append_decode, prefill): the entry points' addresses */
static PyObject* bind(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void* p[4];
  if (!count(n, 4)) return NULL;
  for (int i = 0; i < 4; ++i)
    if (!get_ptr(a[i], &p[i])) return NULL;
  *(void**)&f_append = p[0]; *(void**)&f_decode = p[1]; *(void**)&f_append_decode = p[2]; *(void**)&f_prefill = p[3];
  Py_RETURN_NONE;
}

#define FAST(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {FAST(append), FAST(decode), FAST(append_decode), FAST(prefill), FAST(bind), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_call", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__call(void) {
  s_is_cuda = PyUnicode_InternFromString("is_cuda");
  s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_nbytes = PyUnicode_InternFromString("nbytes");
  return PyModule_Create(&module);
}
