/* Calls of the C ABI (include/aqt.h) from Python with plain integers for arguments.
 *
 * A call of an entry point through ctypes spends 8.6 us of host time turning its twenty arguments
 * into ctypes objects and those into registers, more than the launches behind it (about 2 us each),
 * and small layers are bound by it.  Here an argument is a Python integer (anything int() takes), an
 * address (None is the null pointer) or a float, read by the vector-call convention: 0.5 us.  The interpreter lock is
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

/* The value of a Python integer.  Addresses are unsigned: the low 64 bits of either reading are the same. */
static inline int read_long(PyObject* v, int64_t* out) {
  int overflow = 0;
  *out = PyLong_AsLongLongAndOverflow(v, &overflow);
  if (__builtin_expect(*out != -1 && overflow == 0, 1)) return 1;
  if (overflow > 0) *out = (int64_t)PyLong_AsUnsignedLongLong(v);
  if (overflow < 0) PyErr_SetString(PyExc_OverflowError, "argument out of range");
  return !PyErr_Occurred();
}
/* An integer argument that is none yet: what int() takes, as the ctypes calls do (TypeError for None). */
static int read_number(PyObject* v, int64_t* out) {
  PyObject* n = PyNumber_Long(v);
  if (n == NULL) return 0;
  const int ok = read_long(n, out);
  Py_DECREF(n);
  return ok;
}

/* types: one character per argument, 'p' (address or None), 'i' (integer) or 'f' (float). */
static int read_args(PyObject* const* args, Py_ssize_t nargs, const char* types, Arg* out) {
  Py_ssize_t n = 0;
  for (; types[n] != 0; ++n) {
    if (n >= nargs) break;
    PyObject* v = args[n];
    if (types[n] == 'f') {
      out[n].f = PyFloat_AsDouble(v);
      if (out[n].f == -1.0 && PyErr_Occurred()) return 0;
    } else if (PyLong_Check(v)) {
      if (!read_long(v, &out[n].i)) return 0;
    } else if (types[n] == 'p' && v == Py_None) {
      out[n].i = 0;
    } else if (!read_number(v, &out[n].i)) {
      return 0;
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

ENTRY(quantize, "piiiiiiippp", fn(P(0), I(1), I(2), I(3), N(4), N(5), N(6), N(7), P(8), P(9), P(10)))
ENTRY(qmatmul, "ppippppifiiiiiipippip",
      fn(P(0), P(1), N(2), P(3), P(4), P(5), P(6), I(7), F(8), I(9), I(10), I(11), N(12), N(13), N(14), P(15), I(16), P(17), P(18), Z(19), P(20)))
ENTRY(qmatmul_with_plan, "pppippppifiiiiiipippip",
      fn(P(0), P(1), P(2), N(3), P(4), P(5), P(6), P(7), I(8), F(9), I(10), I(11), I(12), N(13), N(14), N(15), P(16), I(17), P(18), P(19), Z(20), P(21)))
ENTRY(qmatmul_requant, "ppippppifiiiiiiiiipppipip",
      fn(P(0), P(1), N(2), P(3), P(4), P(5), P(6), I(7), F(8), I(9), I(10), I(11), N(12), N(13), N(14), N(15), N(16), N(17), P(18), P(19),
         P(20), I(21), P(22), Z(23), P(24)))
ENTRY(qmatmul_requant_from, "ippippp" "iiiiiii" "ppp" "ipip",
      fn(I(0), P(1), P(2), N(3), P(4), P(5), P(6), I(7), I(8), I(9), N(10), N(11), N(12), N(13), P(14), P(15), P(16), I(17), P(18), Z(19), P(20)))
ENTRY(linear_fwd, "pippppifiiiiiiiipipip",
      fn(P(0), I(1), P(2), P(3), P(4), P(5), I(6), F(7), I(8), I(9), I(10), N(11), N(12), N(13), N(14), N(15), P(16), I(17), P(18), Z(19), P(20)))
ENTRY(linear_fwd_weight_only, "pippppifiiiiiipipip",
      fn(P(0), I(1), P(2), P(3), P(4), P(5), I(6), F(7), I(8), I(9), I(10), N(11), N(12), N(13), P(14), I(15), P(16), Z(17), P(18)))
ENTRY(linear_bwd, "pippiippiiiipipippip",
      fn(P(0), I(1), P(2), P(3), N(4), N(5), P(6), P(7), N(8), I(9), I(10), I(11), P(12), I(13), P(14), I(15), P(16), P(17), Z(18), P(19)))
ENTRY(ffn_fwd, "pipppipppiiiiiiipipip",
      fn(P(0), N(1), P(2), P(3), P(4), N(5), P(6), P(7), P(8), N(9), I(10), I(11), I(12), N(13), N(14), N(15), P(16), N(17), P(18), Z(19), P(20)))

/* ---- chains: the layers' addresses and sizes are read from the QuantLinear objects on every call */
static __typeof__(&aqt_chain_fwd) p_chain_fwd = NULL;
static PyObject *s_wq, *s_s_w, *s_bias, *s_spec, *s_N, *s_K, *s_act, *s_bits_w, *s_bits_a, *s_data_ptr;

static int attr_int(PyObject* o, PyObject* name, int32_t* out) {
  PyObject* v = PyObject_GetAttr(o, name);
  if (v == NULL) return 0;
  const long n = PyLong_AsLong(v);
  Py_DECREF(v);
  if (n == -1 && PyErr_Occurred()) return 0;
  *out = (int32_t)n;
  return 1;
}
static int attr_addr(PyObject* o, PyObject* name, void** out) {
  PyObject* v = PyObject_GetAttr(o, name);
  if (v == NULL) return 0;
  *out = NULL;
  if (v != Py_None) {
    PyObject* a = PyObject_CallMethodNoArgs(v, s_data_ptr);
    if (a != NULL) {
      *out = PyLong_AsVoidPtr(a);
      Py_DECREF(a);
    }
  }
  Py_DECREF(v);
  return !PyErr_Occurred();
}
static int read_layer(PyObject* layer, aqt_chain_layer* l) {
  PyObject* spec = PyObject_GetAttr(layer, s_spec);
  if (spec == NULL) return 0;
  const int ok = attr_int(spec, s_N, &l->N) && attr_int(spec, s_K, &l->K) && attr_int(spec, s_act, &l->act) &&
                 attr_int(spec, s_bits_w, &l->bits_w) && attr_int(spec, s_bits_a, &l->bits_a) && attr_addr(layer, s_wq, (void**)&l->wq) &&
                 attr_addr(layer, s_s_w, (void**)&l->s_w) && attr_addr(layer, s_bias, (void**)&l->bias);
  Py_DECREF(spec);
  l->y = NULL;
  l->ldy = 0;
  l->flags = 0;
  l->residual_scale = 1.0f;
  l->reserved = 0;
  return ok;
}

/* chain_ffn(x, ldx, M, first layer, second layer, y, ldy, rounding, stream) */
static PyObject* w_chain_ffn(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {
  Arg a[9];
  aqt_chain_layer l[2];
  (void)self;
  if (nargs != 9 || p_chain_fwd == NULL) {
    PyErr_SetString(PyExc_TypeError, "chain_ffn: nine arguments, library open");
    return NULL;
  }
  if (!read_args(args, 3, "pii", a) || !read_args(args + 5, 4, "piip", a + 5)) return NULL;
  if (!read_layer(args[3], &l[0]) || !read_layer(args[4], &l[1])) return NULL;
  l[1].y = (float*)P(5);
  l[1].ldy = I(6);
  int status;
  Py_BEGIN_ALLOW_THREADS status = p_chain_fwd(P(0), I(1), I(2), l, 2, N(7), P(8));
  Py_END_ALLOW_THREADS return PyLong_FromLong(status);
}

/* chain_encoder(x, ldx, M, blocks, qkv, ldqkv, out, ldout, rounding, stream): the stand-in dataflow of
 * encoder.py for blocks of ten layers each; q, k, v of the last block are left in qkv, the stack's
 * output in out.  Stacks longer than one call takes go in several, through out. */
static PyObject* w_chain_encoder(PyObject* self, PyObject* const* args, Py_ssize_t nargs) {
  enum { kPerBlock = 10, kBlocks = AQT_CHAIN_MAX_LAYERS / kPerBlock };
  Arg a[10];
  aqt_chain_layer l[kBlocks * kPerBlock];
  (void)self;
  if (nargs != 10 || p_chain_fwd == NULL || !PyList_Check(args[3])) {
    PyErr_SetString(PyExc_TypeError, "chain_encoder: ten arguments, the fourth a list of blocks, library open");
    return NULL;
  }
  if (!read_args(args, 3, "pii", a) || !read_args(args + 4, 6, "pipiip", a + 4)) return NULL;
  const Py_ssize_t n_blocks = PyList_GET_SIZE(args[3]);
  const float* x = (const float*)P(0);
  int64_t ldx = I(1);
  int status = AQT_OK;
  for (Py_ssize_t b0 = 0; b0 < n_blocks && status == AQT_OK; b0 += kBlocks) {
    const Py_ssize_t b1 = b0 + kBlocks < n_blocks ? b0 + kBlocks : n_blocks;
    for (Py_ssize_t b = b0; b < b1; ++b) {
      PyObject* block = PyList_GetItem(args[3], b);
      if (block == NULL || !PyList_Check(block) || PyList_GET_SIZE(block) != kPerBlock) return PyLong_FromLong(AQT_ERR_UNSUPPORTED);
      aqt_chain_layer* q = l + (b - b0) * kPerBlock;
      for (int i = 0; i < kPerBlock; ++i)
        if (!read_layer(PyList_GET_ITEM(block, i), q + i)) return NULL;
      q[1].flags = q[5].flags = q[7].flags = q[9].flags = AQT_CHAIN_ADD;
      q[1].residual_scale = q[9].residual_scale = 0.5f;
      q[2].flags = q[3].flags = AQT_CHAIN_SIDE;
      float* qkv = (float*)P(4);
      for (int i = 2; i < 5; ++i) {
        q[i].y = qkv;
        q[i].ldy = I(5);
        qkv += q[i].N;
      }
    }
    aqt_chain_layer* end = l + (b1 - b0) * kPerBlock - 1;
    end->y = (float*)P(6);
    end->ldy = I(7);
    const int n = (int)(b1 - b0) * kPerBlock;
    Py_BEGIN_ALLOW_THREADS status = p_chain_fwd(x, ldx, I(2), l, n, N(8), P(9));
    Py_END_ALLOW_THREADS x = (const float*)P(6);
    ldx = I(7);
  }
  return PyLong_FromLong(status);
}

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
  RESOLVE(qmatmul_requant_from)
  RESOLVE(linear_fwd)
  RESOLVE(linear_fwd_weight_only)
  RESOLVE(linear_bwd)
  RESOLVE(ffn_fwd)
  RESOLVE(qmatmul_with_plan)
  RESOLVE(workspace_bytes)
  RESOLVE(chain_fwd)
  Py_RETURN_NONE;
}

#define METHOD(NAME) {#NAME, (PyCFunction)(void (*)(void))w_##NAME, METH_FASTCALL, "aqt_" #NAME " (include/aqt.h)"}
static PyMethodDef methods[] = {{"open", w_open, METH_O, "Resolve the entry points in the library at this path."},
                                METHOD(quantize),
                                METHOD(qmatmul),
                                METHOD(qmatmul_requant),
                                METHOD(qmatmul_requant_from),
                                METHOD(linear_fwd),
                                METHOD(linear_fwd_weight_only),
                                METHOD(linear_bwd),
                                METHOD(ffn_fwd),
                                METHOD(qmatmul_with_plan),
                                METHOD(workspace_bytes),
                                METHOD(chain_ffn),
                                METHOD(chain_encoder),
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__fastcall(void) {
#define NAME(v, text) \
  v = PyUnicode_InternFromString(text); \
  if (v == NULL) return NULL;
  NAME(s_wq, "wq") NAME(s_s_w, "s_w") NAME(s_bias, "bias") NAME(s_spec, "spec") NAME(s_N, "N") NAME(s_K, "K")
  NAME(s_act, "act") NAME(s_bits_w, "bits_w") NAME(s_bits_a, "bits_a") NAME(s_data_ptr, "data_ptr")
  return PyModule_Create(&module);
}
