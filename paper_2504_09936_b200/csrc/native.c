// The calls a serving loop makes for every token, from Python objects straight to the C ABI: parameter and cache structs
// through the buffer protocol, tensors through data_ptr().  The same calls through ctypes cost 4.5 us of host time each (13
// arguments converted one by one), more than the launch itself and more than a small decode step takes on the device.
// The functions return the ABI's status code; binding.py turns it into an exception.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "keepkv.h"

static PyObject *s_data_ptr, *s_numel;

// The struct behind a ctypes.Structure of the given size.
static int struct_at(PyObject *o, size_t size, void *to) {
  Py_buffer v;
  if (PyObject_GetBuffer(o, &v, PyBUF_SIMPLE)) return 0;
  const int ok = (size_t)v.len == size;
  if (ok) memcpy(to, v.buf, size);
  PyBuffer_Release(&v);
  if (!ok) PyErr_SetString(PyExc_TypeError, "keepkv_params and keepkv_cache structs expected");
  return ok;
}
// A method without arguments that returns an address or a size.
static int ask(PyObject *o, PyObject *method, uint64_t *to) {
  PyObject *r = PyObject_CallMethodNoArgs(o, method);
  if (!r) return 0;
  *to = PyLong_AsUnsignedLongLong(r);
  Py_DECREF(r);
  return !(*to == (uint64_t)-1 && PyErr_Occurred());
}
static int tensor_at(PyObject *o, void **to) {
  uint64_t v = 0;
  if (o != Py_None && !ask(o, s_data_ptr, &v)) return 0;
  *to = (void *)(uintptr_t)v;
  return 1;
}
static int stream_of(PyObject *o, void **to) {
  *to = PyLong_AsVoidPtr(o);
  return !(*to == NULL && PyErr_Occurred());
}
static int count(const char *name, Py_ssize_t n, Py_ssize_t want) {
  if (n != want) PyErr_Format(PyExc_TypeError, "%s takes %zd arguments, %zd given", name, want, n);
  return n == want;
}

// (params, cache, k_new, v_new, status, stream)
static PyObject *append(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  keepkv_params p;
  keepkv_cache c;
  void *kn, *vn, *st, *stream;
  if (!count("append", n, 6) || !struct_at(a[0], sizeof p, &p) || !struct_at(a[1], sizeof c, &c) || !tensor_at(a[2], &kn) ||
      !tensor_at(a[3], &vn) || !tensor_at(a[4], &st) || !stream_of(a[5], &stream))
    return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = keepkv_append(&p, &c, kn, vn, (int32_t *)st, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

// (params, cache, q, out, lse or None, update_scores, ws, status, stream)
static PyObject *decode_attention(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  keepkv_params p;
  keepkv_cache c;
  void *q, *out, *lse, *ws, *st, *stream;
  uint64_t ws_bytes;
  int update;
  if (!count("decode_attention", n, 9) || !struct_at(a[0], sizeof p, &p) || !struct_at(a[1], sizeof c, &c) ||
      !tensor_at(a[2], &q) || !tensor_at(a[3], &out) || !tensor_at(a[4], &lse) || (update = PyObject_IsTrue(a[5])) < 0 ||
      !tensor_at(a[6], &ws) || !ask(a[6], s_numel, &ws_bytes) || !tensor_at(a[7], &st) || !stream_of(a[8], &stream))
    return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = keepkv_decode_attention(&p, &c, q, out, (float *)lse, update, ws, ws_bytes, (int32_t *)st, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

// (params, cache, q, k_new, v_new, out, lse or None, update_scores, ws, status, stream)
static PyObject *decode_step(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  keepkv_params p;
  keepkv_cache c;
  void *q, *kn, *vn, *out, *lse, *ws, *st, *stream;
  uint64_t ws_bytes;
  int update;
  if (!count("decode_step", n, 11) || !struct_at(a[0], sizeof p, &p) || !struct_at(a[1], sizeof c, &c) ||
      !tensor_at(a[2], &q) || !tensor_at(a[3], &kn) || !tensor_at(a[4], &vn) || !tensor_at(a[5], &out) ||
      !tensor_at(a[6], &lse) || (update = PyObject_IsTrue(a[7])) < 0 || !tensor_at(a[8], &ws) ||
      !ask(a[8], s_numel, &ws_bytes) || !tensor_at(a[9], &st) || !stream_of(a[10], &stream))
    return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = keepkv_decode_step(&p, &c, q, kn, vn, out, (float *)lse, update, ws, ws_bytes, (int32_t *)st, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

// (params, sequence of caches, q_host, k_new_host, v_new_host, out_host, q_dev, k_new_dev, v_new_dev, out_dev,
//  update_scores, ws, status, stream)
static PyObject *decode_step_host_layers(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  keepkv_params p;
  void *t[8], *ws, *st, *stream;
  uint64_t ws_bytes;
  int update;
  if (!count("decode_step_host_layers", n, 14) || !struct_at(a[0], sizeof p, &p)) return NULL;
  for (int i = 0; i < 8; ++i)
    if (!tensor_at(a[2 + i], &t[i])) return NULL;
  if ((update = PyObject_IsTrue(a[10])) < 0 || !tensor_at(a[11], &ws) || !ask(a[11], s_numel, &ws_bytes) ||
      !tensor_at(a[12], &st) || !stream_of(a[13], &stream))
    return NULL;
  PyObject *seq = PySequence_Fast(a[1], "a sequence of caches expected");
  if (!seq) return NULL;
  const Py_ssize_t layers = PySequence_Fast_GET_SIZE(seq);
  keepkv_cache *c = PyMem_Malloc(sizeof *c * (layers > 0 ? layers : 1));
  int ok = c != NULL;
  if (!ok) PyErr_NoMemory();
  for (Py_ssize_t l = 0; ok && l < layers; ++l) ok = struct_at(PySequence_Fast_GET_ITEM(seq, l), sizeof *c, &c[l]);
  Py_DECREF(seq);
  int rc = 0;
  if (ok) {
    Py_BEGIN_ALLOW_THREADS
    rc = keepkv_decode_step_host_layers(&p, c, (int32_t)layers, t[0], t[1], t[2], t[3], t[4], t[5], t[6], t[7], update, ws,
                                        ws_bytes, (int32_t *)st, stream);
    Py_END_ALLOW_THREADS
  }
  PyMem_Free(c);
  return ok ? PyLong_FromLong(rc) : NULL;
}

#define FN(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {FN(append), FN(decode_attention), FN(decode_step), FN(decode_step_host_layers),
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", NULL, -1, methods};

PyMODINIT_FUNC PyInit__native(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_numel = PyUnicode_InternFromString("numel");
  return s_data_ptr && s_numel ? PyModule_Create(&module) : NULL;
}
