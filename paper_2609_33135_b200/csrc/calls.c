/* The C ABI's entry points of a serving step as Python callables.
 *
 * ctypes spends 1.8 us on a call of fifteen arguments, as much as a kernel launch, and a decode step makes three such calls.  These
 * take the same arguments (pointers as integers or None and, for the packed structures, bytes) in 0.3 us.  bind(name, address) returns
 * the callable of an entry point of a loaded library; the GIL is released while the library runs, as ctypes does. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "../../include/mpfa.h"

typedef union {
  void *p;
  int i;
  float f;
  size_t z;
} value;

/* One character per argument: p pointer, i int, f float, z size_t. */
static int convert(const char *name, const char *kinds, PyObject *const *a, Py_ssize_t n, value *v) {
  if (n != (Py_ssize_t)strlen(kinds)) {
    PyErr_Format(PyExc_TypeError, "%s takes %zd arguments (%zd given)", name, (Py_ssize_t)strlen(kinds), n);
    return 0;
  }
  for (Py_ssize_t k = 0; k < n; ++k) {
    if (kinds[k] == 'p') {
      v[k].p = a[k] == Py_None ? NULL : PyBytes_Check(a[k]) ? (void *)PyBytes_AS_STRING(a[k]) : PyLong_AsVoidPtr(a[k]);
      if (!v[k].p && PyErr_Occurred()) return 0;
    } else if (kinds[k] == 'i') {
      const long x = PyLong_AsLong(a[k]);
      if (x == -1 && PyErr_Occurred()) return 0;
      if (x != (int)x) {
        PyErr_Format(PyExc_OverflowError, "%s: argument %zd does not fit an int", name, k + 1);
        return 0;
      }
      v[k].i = (int)x;
    } else if (kinds[k] == 'f') {
      const double x = PyFloat_AsDouble(a[k]);
      if (x == -1.0 && PyErr_Occurred()) return 0;
      v[k].f = (float)x;
    } else {
      v[k].z = PyLong_AsSize_t(a[k]);
      if (v[k].z == (size_t)-1 && PyErr_Occurred()) return 0;
    }
  }
  return 1;
}

#define ENTRY(NAME, KINDS, ...)                                                        \
  static PyObject *call_##NAME(PyObject *self, PyObject *const *a, Py_ssize_t n) {     \
    value v[sizeof(KINDS)];                                                            \
    mpfa_status rc;                                                                    \
    if (!convert(#NAME, KINDS, a, n, v)) return NULL;                                  \
    __typeof__(&NAME) f = (__typeof__(&NAME))PyLong_AsVoidPtr(self);                   \
    Py_BEGIN_ALLOW_THREADS                                                             \
    rc = f(__VA_ARGS__);                                                               \
    Py_END_ALLOW_THREADS                                                               \
    return PyLong_FromLong((long)rc);                                                  \
  }

ENTRY(mpfa_quantize_qk, "ppiiiiiipppppzp", v[0].p, v[1].p, v[2].i, v[3].i, v[4].i, v[5].i, v[6].i, v[7].i, v[8].p, v[9].p, v[10].p, v[11].p,
      v[12].p, v[13].z, v[14].p)
ENTRY(mpfa_quantize_qkv, "pppiiiiiifppppppzp", v[0].p, v[1].p, v[2].p, v[3].i, v[4].i, v[5].i, v[6].i, v[7].i, v[8].i, v[9].f, v[10].p, v[11].p,
      v[12].p, v[13].p, v[14].p, v[15].p, v[16].z, v[17].p)
ENTRY(mpfa_quantize_kv_paged, "ppiiiiipfpppzp", v[0].p, v[1].p, v[2].i, v[3].i, v[4].i, v[5].i, v[6].i, v[7].p, v[8].f, v[9].p, v[10].p, v[11].p,
      v[12].z, v[13].p)
ENTRY(mpfa_append_kv_paged, "ppiiiipfppipp", v[0].p, v[1].p, v[2].i, v[3].i, v[4].i, v[5].i, v[6].p, v[7].f, v[8].p, v[9].p, v[10].i, v[11].p,
      v[12].p)
ENTRY(mpfa_prefill, "pppppfifpppp", v[0].p, v[1].p, v[2].p, v[3].p, v[4].p, v[5].f, v[6].i, v[7].f, v[8].p, v[9].p, v[10].p, v[11].p)
ENTRY(mpfa_prefill_paged, "pppipppffpppp", v[0].p, v[1].p, v[2].p, v[3].i, v[4].p, v[5].p, v[6].p, v[7].f, v[8].f, v[9].p, v[10].p, v[11].p,
      v[12].p)
ENTRY(mpfa_decode, "pppippffpppzpp", v[0].p, v[1].p, v[2].p, v[3].i, v[4].p, v[5].p, v[6].f, v[7].f, v[8].p, v[9].p, v[10].p, v[11].z, v[12].p,
      v[13].p)

#define DEF(NAME) {#NAME, (PyCFunction)(void (*)(void))call_##NAME, METH_FASTCALL, NULL}
static PyMethodDef entries[] = {DEF(mpfa_quantize_qk),     DEF(mpfa_quantize_qkv), DEF(mpfa_quantize_kv_paged), DEF(mpfa_append_kv_paged),
                                DEF(mpfa_prefill), DEF(mpfa_prefill_paged), DEF(mpfa_decode)};

static PyObject *bind(PyObject *module, PyObject *args) {
  const char *name;
  PyObject *address;
  (void)module;
  if (!PyArg_ParseTuple(args, "sO!", &name, &PyLong_Type, &address)) return NULL;
  for (size_t i = 0; i < sizeof(entries) / sizeof(entries[0]); ++i)
    if (strcmp(entries[i].ml_name, name) == 0) return PyCFunction_New(&entries[i], address);
  return PyErr_Format(PyExc_KeyError, "%s", name);
}

static PyMethodDef methods[] = {{"bind", bind, METH_VARARGS, "bind(name, address): the callable of an entry point"}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_mpfa_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__mpfa_calls(void) { return PyModule_Create(&module); }
