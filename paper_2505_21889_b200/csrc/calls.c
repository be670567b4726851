/* Argument marshalling of the per-step calls (CPython extension `_calls`).
 *
 * A decode step takes the GPU a few microseconds, and converting its seventeen arguments in Python and
 * ctypes took the host about as long.  Here a call is one C function: descriptors come as addresses,
 * device memory as anything with a data_ptr() (a torch tensor), as an integer address or None, a plan as a
 * numpy array.  Returns the efim_status as an int; nothing else happens here. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include "efim.h"

static PyObject *s_data_ptr, *s_nbytes;
static PyTypeObject* ndarray; /* numpy.ndarray */

/* address of a numpy array's memory, which the object keeps valid */
static int array_ptr(PyObject* o, void** out) {
  Py_buffer b;
  if (PyObject_GetBuffer(o, &b, PyBUF_STRIDES) != 0) return 0;
  *out = b.buf;
  PyBuffer_Release(&b);
  return 1;
}
/* address of a device tensor, an integer address, a numpy array (over memory that the device can address), or
   NULL for None.  Not of any other object with a buffer: a numpy scalar's is a temporary. */
static int as_ptr(PyObject* o, void** out) {
  if (o == Py_None) {
    *out = NULL;
    return 1;
  }
  if (PyLong_Check(o)) {
    *out = PyLong_AsVoidPtr(o);
    return !(*out == NULL && PyErr_Occurred());
  }
  if (PyObject_TypeCheck(o, ndarray)) return array_ptr(o, out);
  PyObject* r = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (!r) return 0;
  *out = PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return !(*out == NULL && PyErr_Occurred());
}
static int as_i32(PyObject* o, int32_t* out) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) return 0;
  *out = (int32_t)v;
  return 1;
}
static int as_float(PyObject* o, float* out) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) return 0;
  *out = (float)v;
  return 1;
}
/* bytes of an object with an `nbytes`, 0 for None */
static int as_bytes(PyObject* o, size_t* out) {
  *out = 0;
  if (o == Py_None) return 1;
  PyObject* r = PyObject_GetAttr(o, s_nbytes);
  if (!r) return 0;
  *out = PyLong_AsSize_t(r);
  Py_DECREF(r);
  return !(*out == (size_t)-1 && PyErr_Occurred());
}
/* a workspace: device memory whose size the object knows */
static int as_workspace(PyObject* o, void** out, size_t* bytes) {
  if (PyObject_TypeCheck(o, ndarray)) {
    PyErr_SetString(PyExc_TypeError, "the workspace is device memory, not a numpy array");
    return 0;
  }
  return as_ptr(o, out) && as_bytes(o, bytes);
}
/* a plan: host memory, a numpy array or None */
static int as_plan(PyObject* o, void** out, size_t* bytes) {
  *out = NULL;
  *bytes = 0;
  if (o == Py_None) return 1;
  if (!PyObject_TypeCheck(o, ndarray)) {
    PyErr_SetString(PyExc_TypeError, "the plan is a numpy array in host memory");
    return 0;
  }
  return array_ptr(o, out) && as_bytes(o, bytes);
}
static int want(Py_ssize_t n, Py_ssize_t expected) {
  if (n == expected) return 1;
  PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", expected, n);
  return 0;
}
#define PTR(i) as_ptr(a[i], &p[i])
/* a launch can wait for room in the stream's queue: other Python threads go on meanwhile */
#define RETURN_STATUS(call)        \
  do {                             \
    efim_status st_;               \
    Py_BEGIN_ALLOW_THREADS         \
    st_ = (call);                  \
    Py_END_ALLOW_THREADS           \
    return PyLong_FromLong(st_);   \
  } while (0)

/* cache, batch, rope, q, k_new, v_new, status, stream */
static PyObject* kv_append(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void* p[8];
  if (!want(n, 8)) return NULL;
  for (int i = 0; i < 8; ++i)
    if (!PTR(i)) return NULL;
  RETURN_STATUS(efim_kv_append(p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7]));
}

/* cache, batch, q, out, lse, sm_scale, workspace, status, stream, plan or None, lists_resident */
static PyObject* append_prefill_attn(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void* p[11];
  float scale;
  size_t ws, plan_bytes;
  int32_t resident;
  if (!want(n, 11)) return NULL;
  if (!PTR(0) || !PTR(1) || !PTR(2) || !PTR(3) || !PTR(4) || !as_float(a[5], &scale) ||
      !as_workspace(a[6], &p[6], &ws) || !PTR(7) || !PTR(8) || !as_plan(a[9], &p[9], &plan_bytes) ||
      !as_i32(a[10], &resident))
    return NULL;
  if (a[9] == Py_None)
    RETURN_STATUS(efim_append_prefill_attn(p[0], p[1], p[2], p[3], p[4], scale, p[6], ws, p[7], p[8]));
  RETURN_STATUS(efim_append_prefill_attn_planned(p[0], p[1], p[9], plan_bytes, resident, p[2], p[3], p[4], scale,
                                                          p[6], ws, p[7], p[8]));
}

/* cache, batch, rope, q, k_new, v_new, out, lse, sm_scale, plan or None, lists_resident, workspace, status, stream */
static PyObject* append_prefill_step(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void* p[14];
  float scale;
  size_t ws, plan_bytes;
  int32_t resident;
  if (!want(n, 14)) return NULL;
  for (int i = 0; i < 8; ++i)
    if (!PTR(i)) return NULL;
  if (!as_float(a[8], &scale) || !as_plan(a[9], &p[9], &plan_bytes) || !as_i32(a[10], &resident) ||
      !as_workspace(a[11], &p[11], &ws) || !PTR(12) || !PTR(13))
    return NULL;
  RETURN_STATUS(efim_append_prefill_step(p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], scale, p[9], plan_bytes,
                                                  resident, p[11], ws, p[12], p[13]));
}

/* cache, batch, ctx_len, max_ctx_len, block_table, max_pages, q, out, lse, sm_scale, workspace, status, stream */
static PyObject* decode_attn(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void* p[13];
  int32_t batch, max_ctx, max_pages;
  float scale;
  size_t ws;
  if (!want(n, 13)) return NULL;
  if (!PTR(0) || !as_i32(a[1], &batch) || !PTR(2) || !as_i32(a[3], &max_ctx) || !PTR(4) || !as_i32(a[5], &max_pages) ||
      !PTR(6) || !PTR(7) || !PTR(8) || !as_float(a[9], &scale) ||
      !as_workspace(a[10], &p[10], &ws) || !PTR(11) || !PTR(12))
    return NULL;
  RETURN_STATUS(efim_decode_attn(p[0], batch, p[2], max_ctx, p[4], max_pages, p[6], p[7], p[8], scale, p[10], ws,
                                          p[11], p[12]));
}

/* cache, batch, ctx_len, max_ctx_len, block_table, max_pages, rope, q, k_new, v_new, out, lse, sm_scale, workspace,
   status, stream */
static PyObject* decode_step(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void* p[16];
  int32_t batch, max_ctx, max_pages;
  float scale;
  size_t ws;
  if (!want(n, 16)) return NULL;
  if (!PTR(0) || !as_i32(a[1], &batch) || !PTR(2) || !as_i32(a[3], &max_ctx) || !PTR(4) || !as_i32(a[5], &max_pages))
    return NULL;
  for (int i = 6; i < 12; ++i)
    if (!PTR(i)) return NULL;
  if (!as_float(a[12], &scale) || !as_workspace(a[13], &p[13], &ws) || !PTR(14) || !PTR(15)) return NULL;
  RETURN_STATUS(efim_decode_step(p[0], batch, p[2], max_ctx, p[4], max_pages, p[6], p[7], p[8], p[9], p[10], p[11],
                                          scale, p[13], ws, p[14], p[15]));
}

static PyMethodDef methods[] = {
    {"kv_append", (PyCFunction)(void*)kv_append, METH_FASTCALL, NULL},
    {"append_prefill_attn", (PyCFunction)(void*)append_prefill_attn, METH_FASTCALL, NULL},
    {"append_prefill_step", (PyCFunction)(void*)append_prefill_step, METH_FASTCALL, NULL},
    {"decode_attn", (PyCFunction)(void*)decode_attn, METH_FASTCALL, NULL},
    {"decode_step", (PyCFunction)(void*)decode_step, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_nbytes = PyUnicode_InternFromString("nbytes");
  PyObject* numpy = PyImport_ImportModule("numpy");
  if (!s_data_ptr || !s_nbytes || !numpy) return NULL;
  ndarray = (PyTypeObject*)PyObject_GetAttrString(numpy, "ndarray");
  Py_DECREF(numpy);
  if (!ndarray || !PyType_Check(ndarray)) return NULL;
  return PyModule_Create(&module);
}
