/* The call path of the Python binding: converts an entry point's arguments and calls it.
 *
 * Every argument of the C ABI is an integer or a pointer, so one function serves all entry points:
 *     call(address, stream, *args) -> the entry point's return value
 * with args converted by kind -- None: NULL; int: itself; a ctypes structure or array (anything with a buffer): its
 * address; a list or tuple of ints: an int32 array that lives for the call; else a tensor: its data_ptr() -- and the raw
 * stream appended as the last argument (None: the current stream of the current device).
 * What bounds it: interpreter overhead.  ctypes needs about 6 us for a 17-argument call plus 2 us for
 * torch.cuda.current_stream(); short layers are issued at that rate, so a model's step of 32 short layers was bound by
 * it.  Here a call costs about 1 us.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <stdlib.h>

#define MAX_ARGS 28
#define STACK_INTS 512

static PyObject *s_data_ptr, *s_cuda_stream;
static PyObject *f_get_device, *f_raw_stream, *f_current_stream, *f_initialized;
static int g_cuda_ready = 0;

/* torch's functions, looked up on the first use (the module is importable without a GPU) */
static int resolve_torch(void) {
  if (f_raw_stream) return 0;
  PyObject* c = PyImport_ImportModule("torch._C");
  PyObject* cuda = c ? PyImport_ImportModule("torch.cuda") : NULL;
  if (cuda) {
    f_get_device = PyObject_GetAttrString(c, "_cuda_getDevice");
    f_current_stream = PyObject_GetAttrString(cuda, "current_stream");
    f_initialized = PyObject_GetAttrString(cuda, "is_initialized");
    f_raw_stream = PyObject_GetAttrString(c, "_cuda_getCurrentRawStream");
  }
  Py_XDECREF(c);
  Py_XDECREF(cuda);
  return f_get_device && f_current_stream && f_initialized && f_raw_stream ? 0 : -1;
}

static int raw_stream(PyObject* stream, uintptr_t* out) {
  PyObject* v = NULL;
  if (stream != Py_None) {
    v = PyObject_GetAttr(stream, s_cuda_stream);
  } else {
    if (resolve_torch() < 0) return -1;
    if (!g_cuda_ready) {
      PyObject* r = PyObject_CallNoArgs(f_initialized);
      if (!r) return -1;
      g_cuda_ready = r == Py_True;
      Py_DECREF(r);
    }
    if (g_cuda_ready) {
      PyObject* dev = PyObject_CallNoArgs(f_get_device);
      if (!dev) return -1;
      v = PyObject_CallOneArg(f_raw_stream, dev);
      Py_DECREF(dev);
    } else {                                       /* torch has not touched the device yet: its own call sets it up */
      PyObject* s = PyObject_CallNoArgs(f_current_stream);
      if (!s) return -1;
      v = PyObject_GetAttr(s, s_cuda_stream);
      Py_DECREF(s);
    }
  }
  if (!v) return -1;
  *out = (uintptr_t)PyLong_AsUnsignedLongLongMask(v);
  Py_DECREF(v);
  return PyErr_Occurred() ? -1 : 0;
}

typedef long long W;

static int invoke(void* f, W* a) {
  /* System V x86-64 and AArch64 pass integers and pointers alike, and a callee never looks at surplus ones, so every
   * entry point can be called with the longest argument list */
  return ((int (*)(W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W, W))f)(
      a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], a[13], a[14], a[15], a[16], a[17],
      a[18], a[19], a[20], a[21], a[22], a[23], a[24], a[25], a[26], a[27]);
}

static PyObject* call(PyObject* self, PyObject* const* args, Py_ssize_t n) {
  W a[MAX_ARGS] = {0};
  int32_t small[STACK_INTS];
  int32_t* heap = NULL;
  Py_ssize_t used = 0;
  Py_buffer views[4];
  int n_views = 0, ok = 0, rc = 0;
  (void)self;
  if (n < 2 || n - 1 > MAX_ARGS) {
    PyErr_SetString(PyExc_TypeError, "call(address, stream, *args)");
    return NULL;
  }
  void* f = PyLong_AsVoidPtr(args[0]);
  if (!f) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null entry point");
    return NULL;
  }
  for (Py_ssize_t i = 2; i < n; ++i) {
    PyObject* o = args[i];
    W* dst = &a[i - 2];
    if (o == Py_None) continue;
    if (PyLong_Check(o)) {
      *dst = PyLong_AsLongLong(o);
      if (*dst == -1 && PyErr_Occurred()) goto done;
    } else if (PyObject_CheckBuffer(o)) {
      if (n_views == 4) { PyErr_SetString(PyExc_TypeError, "too many buffers"); goto done; }
      if (PyObject_GetBuffer(o, &views[n_views], PyBUF_WRITABLE) < 0) goto done;
      *dst = (W)(intptr_t)views[n_views++].buf;
    } else if (PyList_CheckExact(o) || PyTuple_CheckExact(o)) {
      const Py_ssize_t len = PySequence_Fast_GET_SIZE(o);
      int32_t* buf;
      if (used + len <= STACK_INTS) {
        buf = small + used;
        used += len;
      } else {
        if (heap) { PyErr_SetString(PyExc_TypeError, "too many long lists"); goto done; }
        heap = (int32_t*)malloc((size_t)len * sizeof(int32_t));
        if (!heap) { PyErr_NoMemory(); goto done; }
        buf = heap;
      }
      for (Py_ssize_t j = 0; j < len; ++j) {
        PyObject* e = PySequence_Fast_GET_ITEM(o, j);
        long x = PyLong_AsLong(e);
        if (x == -1 && PyErr_Occurred()) {               /* not an int: what int(e) makes of it */
          PyErr_Clear();
          PyObject* as_int = PyNumber_Long(e);
          if (!as_int) goto done;
          x = PyLong_AsLong(as_int);
          Py_DECREF(as_int);
          if (x == -1 && PyErr_Occurred()) goto done;
        }
        buf[j] = (int32_t)x;
      }
      *dst = (W)(intptr_t)buf;
    } else {
      PyObject* v = PyObject_CallMethodNoArgs(o, s_data_ptr);
      if (!v) goto done;
      *dst = (W)PyLong_AsUnsignedLongLongMask(v);
      Py_DECREF(v);
      if (PyErr_Occurred()) goto done;
    }
  }
  {
    uintptr_t st = 0;
    if (raw_stream(args[1], &st) < 0) goto done;
    a[n - 2] = (W)st;
  }
  Py_BEGIN_ALLOW_THREADS
  rc = invoke(f, a);
  Py_END_ALLOW_THREADS
  ok = 1;
done:
  while (n_views > 0) PyBuffer_Release(&views[--n_views]);
  free(heap);
  return ok ? PyLong_FromLong(rc) : NULL;
}

static PyMethodDef methods[] = {
    {"call", (PyCFunction)(void (*)(void))call, METH_FASTCALL, "call(address, stream, *args) -> int"},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_slkv_call", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__slkv_call(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  if (!s_data_ptr || !s_cuda_stream) return NULL;
  return PyModule_Create(&module);
}
