// Argument marshalling of the binding's per-step calls, in C: a layer-step is six calls of a few microseconds of launch
// work each, and ctypes spent as much again on turning tensors, streams and integers into C arguments (6 us per call
// against 0.6 here).  make(address, signature) returns a Python callable for one C entry point; the signature has one
// character per argument:
//   i  integer            f  fp32 number        p  device / host buffer or None (tensor, or what the fallback accepts)
//   s  stream or None (the current one)
// The call runs without the interpreter lock (it may wait for the GPU) and returns the C function's int.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#define MAX_ARGS 16

typedef struct {
  void* fn;
  int n;
  char sig[MAX_ARGS + 1];
} Entry;

static PyTypeObject* tensor_type;              // torch.Tensor
static PyObject *ptr_fallback, *stream_fallback;  // binding._ptr, binding._stream
static PyObject *raw_stream, *raw_device;      // torch's raw getters, once CUDA is initialised
static PyObject *s_data_ptr, *s_is_contiguous, *s_cuda_stream;

// Integer and pointer arguments travel in registers and stack words, fp32 arguments in vector registers of their own, so
// one prototype serves every entry point (x86-64 System V; surplus words are ignored by the callee).
typedef int (*Fn)(uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t,
                  uint64_t, float, float);
#if !defined(__x86_64__)
#error "pycall.c relies on the x86-64 System V calling convention"
#endif

static int to_u64(PyObject* o, uint64_t* out) {
  if (o == Py_None) {
    *out = 0;
    return 0;
  }
  PyObject* i = PyNumber_Index(o);
  if (!i) return -1;
  *out = (uint64_t)PyLong_AsUnsignedLongLongMask(i);
  Py_DECREF(i);
  return PyErr_Occurred() ? -1 : 0;
}
static int take_u64(PyObject* o, uint64_t* out) {  // steals o
  if (!o) return -1;
  int r = to_u64(o, out);
  Py_DECREF(o);
  return r;
}

static int to_pointer(PyObject* o, uint64_t* out) {
  if (o == Py_None) {
    *out = 0;
    return 0;
  }
  if (tensor_type && PyObject_TypeCheck(o, tensor_type)) {
    PyObject* c = PyObject_CallMethodNoArgs(o, s_is_contiguous);
    if (!c) return -1;
    const int yes = c == Py_True;
    Py_DECREF(c);
    if (yes) return take_u64(PyObject_CallMethodNoArgs(o, s_data_ptr), out);
  }
  return take_u64(PyObject_CallOneArg(ptr_fallback, o), out);
}

static int to_stream(PyObject* o, uint64_t* out) {
  if (o == Py_None) {
    if (!raw_stream) return take_u64(PyObject_CallOneArg(stream_fallback, Py_None), out);
    PyObject* dev = PyObject_CallNoArgs(raw_device);
    if (!dev) return -1;
    PyObject* s = PyObject_CallOneArg(raw_stream, dev);
    Py_DECREF(dev);
    return take_u64(s, out);
  }
  if (PyLong_Check(o)) return to_u64(o, out);
  return take_u64(PyObject_GetAttr(o, s_cuda_stream), out);
}

static PyObject* entry_call(PyObject* self, PyObject* const* args, Py_ssize_t n) {
  const Entry* e = (const Entry*)PyCapsule_GetPointer(self, "entry");
  if (!e) return NULL;
  if (n != e->n) return PyErr_Format(PyExc_TypeError, "expected %d arguments, got %zd", e->n, n);
  uint64_t a[14] = {0};
  float f[2] = {0.f, 0.f};
  int na = 0, nf = 0;
  for (int i = 0; i < e->n; ++i) {
    int r = 0;
    switch (e->sig[i]) {
      case 'i': r = args[i] == Py_None ? (PyErr_SetString(PyExc_TypeError, "an integer is required"), -1) : to_u64(args[i], &a[na++]); break;
      case 'p': r = to_pointer(args[i], &a[na++]); break;
      case 's': r = to_stream(args[i], &a[na++]); break;
      default: {
        const double d = PyFloat_AsDouble(args[i]);
        if (d == -1.0 && PyErr_Occurred()) r = -1;
        f[nf++] = (float)d;
      }
    }
    if (r < 0) return NULL;
  }
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = ((Fn)e->fn)(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], a[13], f[0], f[1]);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

static PyMethodDef entry_def = {"entry", (PyCFunction)(void (*)(void))entry_call, METH_FASTCALL, NULL};

static void entry_free(PyObject* cap) { PyMem_Free(PyCapsule_GetPointer(cap, "entry")); }

static PyObject* make(PyObject* self, PyObject* args) {
  unsigned long long addr;
  const char* sig;
  (void)self;
  if (!PyArg_ParseTuple(args, "Ks", &addr, &sig)) return NULL;
  int n = 0, nf = 0;
  for (; sig[n]; ++n) {
    if (n >= MAX_ARGS || !strchr("ifps", sig[n])) return PyErr_Format(PyExc_ValueError, "bad signature %s", sig);
    nf += sig[n] == 'f';
  }
  if (!addr || nf > 2 || n - nf > 14) return PyErr_Format(PyExc_ValueError, "bad entry point or signature %s", sig);
  Entry* e = (Entry*)PyMem_Malloc(sizeof(Entry));
  if (!e) return PyErr_NoMemory();
  e->fn = (void*)(uintptr_t)addr;
  e->n = n;
  strcpy(e->sig, sig);
  PyObject* cap = PyCapsule_New(e, "entry", entry_free);
  if (!cap) {
    PyMem_Free(e);
    return NULL;
  }
  PyObject* f = PyCFunction_New(&entry_def, cap);
  Py_DECREF(cap);
  return f;
}

static void keep(PyObject** slot, PyObject* o) {
  Py_XINCREF(o == Py_None ? NULL : o);
  Py_XSETREF(*slot, o == Py_None ? NULL : o);
}

// setup(ptr_fallback, stream_fallback, tensor type or None, raw stream getter or None, raw device getter or None)
static PyObject* setup(PyObject* self, PyObject* args) {
  PyObject *pf, *sf, *tt, *rs, *rd;
  (void)self;
  if (!PyArg_ParseTuple(args, "OOOOO", &pf, &sf, &tt, &rs, &rd)) return NULL;
  if (tt != Py_None && !PyType_Check(tt)) return PyErr_Format(PyExc_TypeError, "a type is required");
  keep(&ptr_fallback, pf);
  keep(&stream_fallback, sf);
  keep((PyObject**)&tensor_type, tt);
  keep(&raw_device, rd);
  keep(&raw_stream, rs);
  Py_RETURN_NONE;
}

static PyMethodDef methods[] = {{"make", make, METH_VARARGS, NULL}, {"setup", setup, METH_VARARGS, NULL}, {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pycall(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  if (!s_data_ptr || !s_is_contiguous || !s_cuda_stream) return NULL;
  return PyModule_Create(&module);
}
