// Python -> C ABI calls without ctypes: call(address, kinds, arg, ...) turns its arguments into those of a C function returning
// la_status, and calls it.
//
// Every argument of the C ABI is an integer or a pointer, so each goes into one 64-bit slot (x86-64 System V: an int is read
// from the slot's low half).  kinds has a letter for each:
//   t  tensor        its address, NULL for None; refused with ValueError unless it is a contiguous CUDA tensor
//   i  integer       its value
//   s  shape         the address of a structure of the type given to bind
//   h  host memory   the address of a ctypes array, or the address itself
//   r  stream        what the function given to bind makes of it, asked when the arguments before it have been accepted
// A decode step spends longer in argument conversion than its kernel runs: through ctypes and Python-level checks a call costs
// 5 us before the launch, this way 2.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#define MAX_ARGS 24

static PyObject *s_is_cuda, *s_is_contiguous, *s_data_ptr, *stream_of;
static PyTypeObject *shape_type, *ctypes_array;

// 1: *out holds the slot; 0: an exception is set.
static int slot(char kind, PyObject* a, uint64_t* out) {
  if (kind == 's' || (kind == 'h' && !PyLong_Check(a))) {
    PyTypeObject* const type = kind == 's' ? shape_type : ctypes_array;
    if (!type || !PyObject_TypeCheck(a, type)) {
      PyErr_Format(PyExc_TypeError, "%s is expected, not %.100s", kind == 's' ? "a shape" : "a ctypes array", Py_TYPE(a)->tp_name);
      return 0;
    }
    Py_buffer view;
    if (PyObject_GetBuffer(a, &view, PyBUF_SIMPLE) != 0) return 0;
    *out = (uint64_t)(uintptr_t)view.buf;
    PyBuffer_Release(&view);  // (the caller holds the object)
    return 1;
  }
  if (kind == 'r') {
    PyObject* const x = stream_of ? PyObject_CallOneArg(stream_of, a) : NULL;
    if (!x) {
      if (!stream_of) PyErr_SetString(PyExc_RuntimeError, "bind has not been called");
      return 0;
    }
    const int ok = slot('i', x, out);
    Py_DECREF(x);
    return ok;
  }
  if (kind != 't') {
    if (!PyLong_Check(a)) {
      PyErr_Format(PyExc_TypeError, "an integer is expected, not %.100s", Py_TYPE(a)->tp_name);
      return 0;
    }
    *out = PyLong_AsUnsignedLongLongMask(a);
    return !(*out == (uint64_t)-1 && PyErr_Occurred());
  }
  if (a == Py_None) {
    *out = 0;
    return 1;
  }
  PyObject* x = PyObject_GetAttr(a, s_is_cuda);
  if (!x) return 0;
  int ok = PyObject_IsTrue(x);
  Py_DECREF(x);
  if (ok > 0) {
    x = PyObject_CallMethodNoArgs(a, s_is_contiguous);
    if (!x) return 0;
    ok = PyObject_IsTrue(x);
    Py_DECREF(x);
  }
  if (ok < 0) return 0;
  if (!ok) {
    PyErr_SetString(PyExc_ValueError, "tensors must be contiguous CUDA tensors");
    return 0;
  }
  x = PyObject_CallMethodNoArgs(a, s_data_ptr);
  if (!x) return 0;
  *out = PyLong_AsUnsignedLongLong(x);
  Py_DECREF(x);
  return !(*out == (uint64_t)-1 && PyErr_Occurred());
}

typedef int (*Fn)(uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t,
                  uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t, uint64_t);

// Slots past the callee's arguments are not read.
static PyObject* call(PyObject* self, PyObject* const* args, Py_ssize_t n) {
  (void)self;
  Py_ssize_t kinds_n = 0;
  const char* const kinds = n >= 2 && PyUnicode_Check(args[1]) ? PyUnicode_AsUTF8AndSize(args[1], &kinds_n) : NULL;
  if (!kinds || kinds_n != n - 2 || kinds_n > MAX_ARGS) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_TypeError, "call(address, kinds, arg, ...): a letter for each of up to 24 arguments");
    return NULL;
  }
  uint64_t a[MAX_ARGS] = {0}, fn;
  if (!slot('i', args[0], &fn)) return NULL;
  for (Py_ssize_t i = 0; i < kinds_n; ++i)
    if (!slot(kinds[i], args[2 + i], &a[i])) return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS;
  rc = ((Fn)(uintptr_t)fn)(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9], a[10], a[11], a[12], a[13], a[14], a[15], a[16], a[17],
                           a[18], a[19], a[20], a[21], a[22], a[23]);
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(rc);
}

static PyObject* bind(PyObject* self, PyObject* args) {
  (void)self;
  PyObject *type, *f;
  if (!PyArg_ParseTuple(args, "O!O", &PyType_Type, &type, &f)) return NULL;
  Py_INCREF(type);
  Py_XSETREF(shape_type, (PyTypeObject*)type);
  Py_INCREF(f);
  Py_XSETREF(stream_of, f);
  Py_RETURN_NONE;
}

static PyMethodDef methods[] = {{"bind", bind, METH_VARARGS, "bind(type of a shape, function that gives a stream's handle)"},
                                {"call", (PyCFunction)(void (*)(void))call, METH_FASTCALL, "call(address, kinds, arg, ...) -> status"},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_la_call", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__la_call(void) {
  s_is_cuda = PyUnicode_InternFromString("is_cuda");
  s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  if (!s_is_cuda || !s_is_contiguous || !s_data_ptr) return NULL;
  PyObject* const ctypes = PyImport_ImportModule("ctypes");
  if (!ctypes) return NULL;
  ctypes_array = (PyTypeObject*)PyObject_GetAttrString(ctypes, "Array");
  Py_DECREF(ctypes);
  if (!ctypes_array || !PyType_Check((PyObject*)ctypes_array)) return NULL;
  return PyModule_Create(&module);
}
