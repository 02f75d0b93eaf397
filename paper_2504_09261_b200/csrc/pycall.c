/* Marshalling of the per-step calls from Python, in C: call(address, handle, layer, scale, buffer, ...)
 * calls the entry point at `address` of the C ABI (hack.h) with three to five buffer arguments and
 * returns its status.  A buffer is None, an integer address or an object with a data_ptr() method.
 * The same call through ctypes takes 1.9 us of host time per step against 0.5; a small step keeps the GPU
 * busy for 2 to 3 us, so a caller that enqueues step by step was limited by it. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

static PyObject* data_ptr_name;

static int address_of(PyObject* o, void** out) {
  if (o == Py_None) {
    *out = NULL;
    return 0;
  }
  if (PyLong_Check(o)) {
    *out = PyLong_AsVoidPtr(o);
    return *out == NULL && PyErr_Occurred() ? -1 : 0;
  }
  PyObject* r = PyObject_CallMethodNoArgs(o, data_ptr_name);
  if (!r) return -1;
  *out = PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

static PyObject* call(PyObject* self, PyObject* const* args, Py_ssize_t n) {
  (void)self;
  if (n < 7 || n > 9) {
    PyErr_SetString(PyExc_TypeError, "call(address, handle, layer, scale, 3 to 5 buffers)");
    return NULL;
  }
  void* fn = PyLong_AsVoidPtr(args[0]);
  void* h = PyLong_AsVoidPtr(args[1]);
  const long layer = PyLong_AsLong(args[2]), scale = PyLong_AsLong(args[3]);
  void* p[5] = {NULL, NULL, NULL, NULL, NULL};
  if (PyErr_Occurred()) return NULL;
  for (Py_ssize_t i = 4; i < n; ++i)
    if (address_of(args[i], &p[i - 4])) return NULL;
  int status;
  Py_BEGIN_ALLOW_THREADS
  const int32_t l = (int32_t)layer, k = (int32_t)scale;
  if (n == 7) status = ((int (*)(void*, int32_t, int32_t, void*, void*, void*))fn)(h, l, k, p[0], p[1], p[2]);
  else if (n == 8) status = ((int (*)(void*, int32_t, int32_t, void*, void*, void*, void*))fn)(h, l, k, p[0], p[1], p[2], p[3]);
  else status = ((int (*)(void*, int32_t, int32_t, void*, void*, void*, void*, void*))fn)(h, l, k, p[0], p[1], p[2], p[3], p[4]);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(status);
}

static PyMethodDef methods[] = {{"call", (PyCFunction)(void (*)(void))call, METH_FASTCALL, "call(address, handle, layer, scale, buffers...) -> status"},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_hackcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__hackcall(void) {
  data_ptr_name = PyUnicode_InternFromString("data_ptr");
  return data_ptr_name ? PyModule_Create(&module) : NULL;
}
