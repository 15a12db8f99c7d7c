/* The library's shortest call without the conversions of a foreign-function interface.
 *
 * A dense perturbation of a norm vector is 1.4 us on the device, and the call costs the host more than that: the launch, and
 * 1.2 us for turning nine Python objects into C arguments through ctypes.  Here the same nine objects arrive as a vectorcall
 * array.  The library itself stays free of Python; bind() is given the address of its function. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "agzo.h"

static __typeof__(&agzo_perturb_dense) perturb_dense_at;      /* the header's signature; the symbol itself is not linked */

static PyObject* bind(PyObject* self, PyObject* address) {
  (void)self;
  void* p = PyLong_AsVoidPtr(address);
  if (p == NULL && PyErr_Occurred()) return NULL;
  perturb_dense_at = (__typeof__(perturb_dense_at))p;
  Py_RETURN_NONE;
}

static PyObject* perturb_dense(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  (void)self;
  if (n != 9 || perturb_dense_at == NULL) {
    PyErr_SetString(PyExc_TypeError, "perturb_dense takes nine arguments, after bind()");
    return NULL;
  }
  agzo_ctx* ctx = (agzo_ctx*)PyLong_AsVoidPtr(a[0]);
  void* w = PyLong_AsVoidPtr(a[1]);
  const int64_t elems = PyLong_AsLongLong(a[2]);
  const int dtype = (int)PyLong_AsLong(a[3]);
  const uint64_t seed = PyLong_AsUnsignedLongLongMask(a[4]);
  const uint32_t layer_id = (uint32_t)PyLong_AsUnsignedLongMask(a[5]);
  const float scale = (float)PyFloat_AsDouble(a[6]);
  const float* d_scale = (const float*)PyLong_AsVoidPtr(a[7]);
  void* stream = PyLong_AsVoidPtr(a[8]);
  if (PyErr_Occurred()) return NULL;
  int status;
  Py_BEGIN_ALLOW_THREADS
  status = perturb_dense_at(ctx, w, elems, dtype, seed, layer_id, scale, d_scale, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(status);
}

static PyMethodDef methods[] = {
    {"bind", bind, METH_O, "Address of agzo_perturb_dense."},
    {"perturb_dense", (PyCFunction)(void (*)(void))perturb_dense, METH_FASTCALL, "agzo_perturb_dense; returns its status."},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_agzo_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__agzo_calls(void) { return PyModule_Create(&module); }
