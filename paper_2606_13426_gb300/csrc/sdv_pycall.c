/* sdv_pycall.c - the calls a serving loop makes, without ctypes: converting 25 arguments
 * takes ctypes 4-5 us, longer than the launch of a small call; here it takes under 1 us.
 * Integers (modulo their C type's range, as ctypes takes them), floats and None for NULL are
 * taken; any other object is a TypeError, upon which the binding calls through ctypes.  The GIL
 * is released around the call, and the entry points' addresses come from the binding, which
 * has loaded the library. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "specdiff.h"

typedef int (*verify_fn)(const void *, const void *, const void *, const float *, int64_t, int, int, int64_t, int,
                         uint64_t, int, const int32_t *, const void *, const float *, int, float, int32_t *, void *,
                         float *, float *, uint32_t *, float *, void *, size_t, sdv_stream_t);
typedef int (*ratios_fn)(const void *, const void *, const void *, const float *, int64_t, int, int, int64_t, int,
                         const int32_t *, float *, float *, void *, size_t, sdv_stream_t);

/* An argument; errors are left for PyErr_Occurred. */
static unsigned long long u64(PyObject *o) {
  if (PyLong_Check(o)) return PyLong_AsUnsignedLongLongMask(o);
  PyErr_SetString(PyExc_TypeError, "an integer is required");
  return 0;
}
static void *ptr(PyObject *o) { return o == Py_None ? NULL : (void *)(uintptr_t)u64(o); }
static float f32(PyObject *o) {
  if (PyFloat_Check(o) || PyLong_Check(o)) return (float)PyFloat_AsDouble(o);
  PyErr_SetString(PyExc_TypeError, "a number is required");
  return 0;
}

static PyObject *wrong_count(const char *name, int want, Py_ssize_t got) {
  PyErr_Format(PyExc_TypeError, "%s takes %d arguments (%zd given)", name, want, got);
  return NULL;
}

/* verify(address, the 25 arguments of sdv_verify_ex): its return code. */
static PyObject *verify(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  if (n != 26) return wrong_count("verify", 26, n);
  const verify_fn fn = (verify_fn)ptr(a[0]);
  ++a;
  const void *x = ptr(a[0]), *mq = ptr(a[1]), *mp = ptr(a[2]);
  const float *sigma = ptr(a[3]);
  const int64_t stride = (int64_t)u64(a[4]), d = (int64_t)u64(a[7]);
  const int B = (int)u64(a[5]), L = (int)u64(a[6]), dtype = (int)u64(a[8]), mode = (int)u64(a[10]);
  const uint64_t seed = u64(a[9]);
  const int32_t *L_eff = ptr(a[11]);
  const void *mqb = ptr(a[12]);
  const float *sgb = ptr(a[13]);
  const int residual = (int)u64(a[14]);
  const float omega = f32(a[15]);
  int32_t *acc = ptr(a[16]);
  void *y = ptr(a[17]);
  float *lr = ptr(a[18]), *dn = ptr(a[19]);
  uint32_t *st = ptr(a[20]);
  float *aux = ptr(a[21]);
  void *ws = ptr(a[22]);
  const size_t bytes = (size_t)u64(a[23]);
  const sdv_stream_t stream = ptr(a[24]);
  int rc;
  if (PyErr_Occurred()) return NULL;
  Py_BEGIN_ALLOW_THREADS
  rc = fn(x, mq, mp, sigma, stride, B, L, d, dtype, seed, mode, L_eff, mqb, sgb, residual, omega, acc, y, lr, dn, st,
          aux, ws, bytes, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

/* ratios(address, the 15 arguments of sdv_log_ratios): its return code. */
static PyObject *ratios(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  if (n != 16) return wrong_count("ratios", 16, n);
  const ratios_fn fn = (ratios_fn)ptr(a[0]);
  ++a;
  const void *x = ptr(a[0]), *mq = ptr(a[1]), *mp = ptr(a[2]);
  const float *sigma = ptr(a[3]);
  const int64_t stride = (int64_t)u64(a[4]), d = (int64_t)u64(a[7]);
  const int B = (int)u64(a[5]), L = (int)u64(a[6]), dtype = (int)u64(a[8]);
  const int32_t *L_eff = ptr(a[9]);
  float *lr = ptr(a[10]), *dn = ptr(a[11]);
  void *ws = ptr(a[12]);
  const size_t bytes = (size_t)u64(a[13]);
  const sdv_stream_t stream = ptr(a[14]);
  int rc;
  if (PyErr_Occurred()) return NULL;
  Py_BEGIN_ALLOW_THREADS
  rc = fn(x, mq, mp, sigma, stride, B, L, d, dtype, L_eff, lr, dn, ws, bytes, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {
    {"verify", (PyCFunction)(void (*)(void))verify, METH_FASTCALL, "verify(address, *arguments of sdv_verify_ex)"},
    {"ratios", (PyCFunction)(void (*)(void))ratios, METH_FASTCALL, "ratios(address, *arguments of sdv_log_ratios)"},
    {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_sdvcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__sdvcall(void) { return PyModule_Create(&module); }
