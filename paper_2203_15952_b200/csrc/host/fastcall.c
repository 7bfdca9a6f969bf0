/* Calls of the C ABI (include/aqt.h) from Python with plain integers for arguments.
 *
 * A call of an entry point through ctypes spends 8.6 us of host time turning its twenty arguments
 * into ctypes objects and those into registers, more than the launches behind it (about 2 us each),
 * and small layers are bound by it.  Here an argument is a Python integer (pointers included; None is
 * the null pointer) or float, read by the vector-call convention: 0.5 us.  The interpreter lock is
 * released around the call, as ctypes does.  The library stays the one file libaqt.so: open() resolves
 * its entry points, nothing is linked. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>
#include <stddef.h>
#include <stdint.h>

#include "../../../include/aqt.h"

typedef union {
  int64_t i;
  double f;
} Arg;
#define P(k) ((void*)(intptr_t)a[k].i)
#define I(k) a[k].i
#define N(k) ((int)a[k].i)
#define F(k) ((float)a[k].f)
#define Z(k) ((size_t)a[k].i)

/* types: one character per argument, 'i' (integer, pointer, None) or 'f'. */
static int read_args(PyObject* const* args, Py_ssize_t nargs, const char* types, Arg* out) {
  Py_ssize_t n = 0;
  for (; types[n] != 0; ++n) {
    if (n >= nargs) break;
    PyObject* v = args[n];
    if (types[n] == 'f') {
      out[n].f = PyFloat_AsDouble(v);
      if (out[n].f == -1.0 && PyErr_Occurred()) return 0;
    } else if (v == Py_None) {
      out[n].i = 0;
    } else {
      /* pointers are unsigned: the low 64 bits of either reading are the same */
      int overflow = 0;
      out[n].i = PyLong_AsLongLongAndOverflow(v, &overflow);
      if (overflow > 0) out[n].i = (int64_t)PyLong_AsUnsignedLongLong(v);
      if (overflow < 0) PyErr_SetString(PyExc_OverflowError, "argument out of range");
      if ((out[n].i == -1 || overflow) && PyErr_Occurred()) return 0;
    }
  }
  if (types[n] != 0 || n != nargs) {
    PyErr_Format(PyExc_TypeError, "wrong number of arguments: %zd", nargs);
    return 0;
  }
  return 1;
}

/* An entry point: its resolved address, its wrapper.  CALL is the call expression in terms of fn and a[]. */
#define ENTRY(NAME, TYPES, CALL)                                                                  \
  static __typeof__(&aqt_##NAME) p_##NAME = NULL;                                                 \
  static PyObject* w_##NAME(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {            \
    Arg a[sizeof(TYPES)];                                                                         \
    __typeof__(&aqt_##NAME) fn = p_##NAME;                                                        \
    int status;                                                                                   \
    (void)self;                                                                                   \
    if (fn == NULL) {                                                                             \
      PyErr_SetString(PyExc_RuntimeError, "libaqt.so is not open");                               \
      return NULL;                                                                                \
    }                                                                                             \
    if (!read_args(args, nargs, TYPES, a)) return NULL;                                           \
    Py_BEGIN_ALLOW_THREADS status = CALL;                                                         \
    Py_END_ALLOW_THREADS return PyLong_FromLong(status);                                          \
  }

ENTRY(quantize, "iiiiiiiiiii", fn(P(0), I(1), I(2), I(3), N(4), N(5), N(6), N(7), P(8), P(9), P(10)))
ENTRY(qmatmul, "iiiiiiiifiiiiiiiiiiii",
      fn(P(0), P(1), N(2), P(3), P(4), P(5), P(6), I(7), F(8), I(9), I(10), I(11), N(12), N(13), N(14), P(15), I(16), P(17), P(18), Z(19), P(20)))
ENTRY(qmatmul_requant, "iiiiiiiifiiiiiiiiiiiiiiii",
      fn(P(0), P(1), N(2), P(3), P(4), P(5), P(6), I(7), F(8), I(9), I(10), I(11), N(12), N(13), N(14), N(15), N(16), N(17), P(18), P(19),
         P(20), I(21), P(22), Z(23), P(24)))
ENTRY(linear_fwd, "iiiiiiifiiiiiiiiiiiii",
      fn(P(0), I(1), P(2), P(3), P(4), P(5), I(6), F(7), I(8), I(9), I(10), N(11), N(12), N(13), N(14), N(15), P(16), I(17), P(18), Z(19), P(20)))
ENTRY(linear_fwd_weight_only, "iiiiiiifiiiiiiiiiii",
      fn(P(0), I(1), P(2), P(3), P(4), P(5), I(6), F(7), I(8), I(9), I(10), N(11), N(12), N(13), P(14), I(15), P(16), Z(17), P(18)))
ENTRY(linear_bwd, "iiiiiiiiiiiiiiiiiiii",
      fn(P(0), I(1), P(2), P(3), N(4), N(5), P(6), P(7), N(8), I(9), I(10), I(11), P(12), I(13), P(14), I(15), P(16), P(17), Z(18), P(19)))
ENTRY(ffn_fwd, "iiiiiiiiiiiiiiiiiiiii",
      fn(P(0), N(1), P(2), P(3), P(4), N(5), P(6), P(7), P(8), N(9), I(10), I(11), I(12), N(13), N(14), N(15), P(16), N(17), P(18), Z(19), P(20)))

static __typeof__(&aqt_workspace_bytes) p_workspace_bytes = NULL;
static PyObject* w_workspace_bytes(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {
  Arg a[6];
  (void)self;
  if (p_workspace_bytes == NULL) {
    PyErr_SetString(PyExc_RuntimeError, "libaqt.so is not open");
    return NULL;
  }
  if (!read_args(args, nargs, "iiiiii", a)) return NULL;
  return PyLong_FromSize_t(p_workspace_bytes(N(0), I(1), I(2), I(3), N(4), N(5)));
}

static PyObject* w_open(PyObject* self, PyObject* path) {
  (void)self;
  const char* s = PyUnicode_AsUTF8(path);
  if (s == NULL) return NULL;
  void* lib = dlopen(s, RTLD_NOW | RTLD_LOCAL);
  if (lib == NULL) {
    PyErr_SetString(PyExc_ImportError, dlerror());
    return NULL;
  }
#define RESOLVE(NAME)                                                \
  *(void**)&p_##NAME = dlsym(lib, "aqt_" #NAME);                     \
  if (p_##NAME == NULL) {                                            \
    PyErr_SetString(PyExc_ImportError, "missing entry point aqt_" #NAME); \
    return NULL;                                                     \
  }
  RESOLVE(quantize)
  RESOLVE(qmatmul)
  RESOLVE(qmatmul_requant)
  RESOLVE(linear_fwd)
  RESOLVE(linear_fwd_weight_only)
  RESOLVE(linear_bwd)
  RESOLVE(ffn_fwd)
  RESOLVE(workspace_bytes)
  Py_RETURN_NONE;
}

#define METHOD(NAME) {#NAME, (PyCFunction)(void (*)(void))w_##NAME, METH_FASTCALL, "aqt_" #NAME " (include/aqt.h)"}
static PyMethodDef methods[] = {{"open", w_open, METH_O, "Resolve the entry points in the library at this path."},
                                METHOD(quantize),
                                METHOD(qmatmul),
                                METHOD(qmatmul_requant),
                                METHOD(linear_fwd),
                                METHOD(linear_fwd_weight_only),
                                METHOD(linear_bwd),
                                METHOD(ffn_fwd),
                                METHOD(workspace_bytes),
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__fastcall(void) { return PyModule_Create(&module); }
