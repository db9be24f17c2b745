// Python entry of litevar_attn_forward: reads pointers and strides of the four tensors and makes the call.
//
// An eager call of a small step is bound by the host.  Through ctypes the marshalling (four stride tuples into structs, four data
// pointers, a fourteen-argument foreign call) takes 3.3 us of the call's 6.1; here it takes 1 (step 3 of a 256px schedule, one
// image, called from Python).  The library stays a plain C ABI: its function's address comes in as an integer, and nothing of
// torch is compiled in (a tensor is whatever has data_ptr(), stride() and get_device()).
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "litevar.h"

typedef litevar_status_t (*forward_fn)(const litevar_plan_t*, int32_t, int32_t, const void*, const litevar_strides_t*, const void*,
                                       const litevar_strides_t*, const void*, const litevar_strides_t*, void*,
                                       const litevar_strides_t*, void*);

static PyObject *s_data_ptr, *s_stride, *s_get_device;

// Data pointer and strides of a [2B, H, tokens, 64] tensor; 0 with a Python error set when it is something else.
static int read_tensor(PyObject* t, void** ptr, litevar_strides_t* s) {
  PyObject* o = PyObject_CallMethodNoArgs(t, s_data_ptr);
  if (!o) return 0;
  *ptr = PyLong_AsVoidPtr(o);
  Py_DECREF(o);
  if (PyErr_Occurred()) return 0;
  o = PyObject_CallMethodNoArgs(t, s_stride);
  if (!o) return 0;
  if (!PyTuple_Check(o) || PyTuple_GET_SIZE(o) != 4 || PyLong_AsLongLong(PyTuple_GET_ITEM(o, 3)) != 1) {
    Py_DECREF(o);
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "expected [2B, H, tokens, 64] tensors with contiguous head_dim");
    return 0;
  }
  s->batch = PyLong_AsLongLong(PyTuple_GET_ITEM(o, 0));
  s->head = PyLong_AsLongLong(PyTuple_GET_ITEM(o, 1));
  s->token = PyLong_AsLongLong(PyTuple_GET_ITEM(o, 2));
  Py_DECREF(o);
  return !PyErr_Occurred();
}

// forward(address of litevar_attn_forward, plan, step_k, batch_pairs, q, k, v, out, stream, current_stream) -> status.
// stream None: current_stream(device index of q), which returns the raw stream.
static PyObject* forward(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  (void)self;
  if (n != 10) {
    PyErr_SetString(PyExc_TypeError, "forward takes 10 arguments");
    return NULL;
  }
  forward_fn fn = (forward_fn)PyLong_AsVoidPtr(a[0]);
  const litevar_plan_t* plan = (const litevar_plan_t*)PyLong_AsVoidPtr(a[1]);
  const long step_k = PyLong_AsLong(a[2]), batch_pairs = PyLong_AsLong(a[3]);
  if (PyErr_Occurred()) return NULL;
  void* ptr[4];
  litevar_strides_t st[4];
  for (int i = 0; i < 4; ++i)
    if (!read_tensor(a[4 + i], &ptr[i], &st[i])) return NULL;
  PyObject* so = a[8];
  if (so == Py_None) {
    PyObject* dev = PyObject_CallMethodNoArgs(a[4], s_get_device);
    if (!dev) return NULL;
    so = PyObject_CallOneArg(a[9], dev);
    Py_DECREF(dev);
    if (!so) return NULL;
  } else {
    Py_INCREF(so);
  }
  void* stream = PyLong_AsVoidPtr(so);
  Py_DECREF(so);
  if (PyErr_Occurred()) return NULL;
  litevar_status_t status;
  Py_BEGIN_ALLOW_THREADS
  status = fn(plan, (int32_t)step_k, (int32_t)batch_pairs, ptr[0], &st[0], ptr[1], &st[1], ptr[2], &st[2], ptr[3], &st[3], stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong((long)status);
}

static PyMethodDef methods[] = {
    {"forward", (PyCFunction)(void (*)(void))forward, METH_FASTCALL, "litevar_attn_forward on tensors; returns the status"},
    {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_litevar_host", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__litevar_host(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_stride = PyUnicode_InternFromString("stride");
  s_get_device = PyUnicode_InternFromString("get_device");
  if (!s_data_ptr || !s_stride || !s_get_device) return NULL;
  return PyModule_Create(&module);
}
