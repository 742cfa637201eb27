/*
 * Python entry points of the calls a program makes in its inner loop (collectives, send/recv): argument marshalling in C.
 *
 * A collective over 8 ranks takes 16 device pointers and the current stream; collecting them in Python and passing them
 * through ctypes cost 8.7 us of an 11 us call, several times what the library itself needs to launch a short message.  Here a
 * pointer is one method call on the tensor and the arguments go straight to the function of libhoccl.so, whose addresses the
 * binding hands over once (bind), so that there is one image of the library in the process.  The GIL is released during the call.
 *
 * Buffers: objects with a data_ptr() method, integers, or None (a null pointer).  Streams: None (the current torch stream), an
 * object with a cuda_stream attribute, or an integer.  Every function returns the library's result code.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#define MAX_RANKS 64

typedef int (*coll_op_fn)(const void* const*, void* const*, size_t, int, int, void*, void*);
typedef int (*coll_fn)(const void* const*, void* const*, size_t, int, void*, void*);
typedef int (*static_fn)(const void* const*, void* const*, size_t, int, int, int, void*);
typedef int (*pattern_fn)(const void* const*, const size_t*, const size_t*, void* const*, const size_t*, int, void*, void*);
typedef int (*p2p_fn)(void*, size_t, int, int, int, void*, void*);

enum { F_ALLREDUCE, F_REDUCE_SCATTER, F_HOST_ALLREDUCE, F_ALLGATHER, F_ALLTOALL, F_ALLTOALLV, F_SEND, F_RECV, F_STATIC, F_COUNT };
static void* g_fn[F_COUNT];
static PyObject *g_data_ptr, *g_cuda_stream;          /* interned attribute names */
static PyObject *g_current_device, *g_current_stream; /* torch's: () -> device index, (device index) -> raw stream */

/* ------------------------------------------------------------------ arguments */

static int as_address(PyObject* o, void** out) {
  if (o == Py_None) {
    *out = NULL;
    return 0;
  }
  PyObject* v;
  if (PyLong_Check(o)) {
    v = Py_NewRef(o);
  } else {
    v = PyObject_CallMethodNoArgs(o, g_data_ptr);
    if (!v && PyErr_ExceptionMatches(PyExc_AttributeError)) {
      PyErr_Clear();
      v = PyNumber_Long(o);
    }
  }
  if (!v) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

/* A sequence of buffers: the first MAX_RANKS of them; entries beyond its length are null, which the library refuses. */
static int as_addresses(PyObject* seq, void** out) {
  PyObject* f = PySequence_Fast(seq, "a sequence of buffers is wanted");
  if (!f) return -1;
  const Py_ssize_t given = PySequence_Fast_GET_SIZE(f), n = given < MAX_RANKS ? given : MAX_RANKS;
  int rc = 0;
  for (Py_ssize_t i = 0; i < n && rc == 0; i++) rc = as_address(PySequence_Fast_GET_ITEM(f, i), &out[i]);
  if (rc == 0) memset(out + n, 0, (size_t)(MAX_RANKS - n) * sizeof(void*));
  Py_DECREF(f);
  return rc;
}

static int as_size(PyObject* o, size_t* out) {
  PyObject* v = PyLong_Check(o) ? Py_NewRef(o) : PyNumber_Long(o);
  if (!v) return -1;
  *out = (size_t)PyLong_AsUnsignedLongLongMask(v);
  Py_DECREF(v);
  return PyErr_Occurred() ? -1 : 0;
}

static int as_int(PyObject* o, int* out) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) return -1;
  *out = (int)v;
  return 0;
}

static int as_dtype(PyObject* o, int* out) {
  if (PyUnicode_Check(o)) {
    if (PyUnicode_CompareWithASCIIString(o, "fp32") == 0) *out = 0;
    else if (PyUnicode_CompareWithASCIIString(o, "bf16") == 0) *out = 1;
    else {
      PyErr_SetObject(PyExc_KeyError, o);
      return -1;
    }
    return 0;
  }
  PyObject* v = PyNumber_Long(o);
  if (!v) return -1;
  const int rc = as_int(v, out);
  Py_DECREF(v);
  return rc;
}

static int as_stream(PyObject* o, void** out) {
  PyObject* v = NULL;
  if (o == Py_None) {
    if (!g_current_stream) {   /* first use: torch may be imported after this module, and CUDA not be up yet */
      PyObject* cuda = PyImport_ImportModule("torch.cuda");
      PyObject* up = cuda ? PyObject_CallMethod(cuda, "init", NULL) : NULL;
      Py_XDECREF(cuda);
      if (!up) return -1;
      Py_DECREF(up);
      PyObject* c = PyImport_ImportModule("torch._C");
      if (!c) return -1;
      g_current_device = PyObject_GetAttrString(c, "_cuda_getDevice");
      g_current_stream = g_current_device ? PyObject_GetAttrString(c, "_cuda_getCurrentRawStream") : NULL;
      Py_DECREF(c);
      if (!g_current_stream) return -1;
    }
    PyObject* dev = PyObject_CallNoArgs(g_current_device);
    if (!dev) return -1;
    v = PyObject_CallOneArg(g_current_stream, dev);
    Py_DECREF(dev);
  } else if (PyLong_Check(o)) {
    v = Py_NewRef(o);
  } else {
    v = PyObject_GetAttr(o, g_cuda_stream);
    if (!v && PyErr_ExceptionMatches(PyExc_AttributeError)) {
      PyErr_Clear();
      v = PyNumber_Long(o);
    }
  }
  if (!v) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

static int n_args(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return 0;
  PyErr_Format(PyExc_TypeError, "%zd arguments, %zd wanted", n, want);
  return -1;
}

/* ------------------------------------------------------------------ calls */

/* (comm, send, recv, count, dtype, op, stream) */
static PyObject* call_with_op(int which, PyObject* const* a, Py_ssize_t n) {
  void *send[MAX_RANKS], *recv[MAX_RANKS], *comm, *stream;
  size_t count;
  int dtype, op, rc;
  if (n_args(n, 7) || as_address(a[0], &comm) || as_addresses(a[1], send) || as_addresses(a[2], recv) || as_size(a[3], &count) ||
      as_dtype(a[4], &dtype) || as_int(a[5], &op) || as_stream(a[6], &stream))
    return NULL;
  Py_BEGIN_ALLOW_THREADS
  rc = ((coll_op_fn)g_fn[which])((const void* const*)send, recv, count, dtype, op, comm, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

/* (comm, send, recv, count, dtype, stream) */
static PyObject* call_without_op(int which, PyObject* const* a, Py_ssize_t n) {
  void *send[MAX_RANKS], *recv[MAX_RANKS], *comm, *stream;
  size_t count;
  int dtype, rc;
  if (n_args(n, 6) || as_address(a[0], &comm) || as_addresses(a[1], send) || as_addresses(a[2], recv) || as_size(a[3], &count) ||
      as_dtype(a[4], &dtype) || as_stream(a[5], &stream))
    return NULL;
  Py_BEGIN_ALLOW_THREADS
  rc = ((coll_fn)g_fn[which])((const void* const*)send, recv, count, dtype, comm, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

/* (comm, buf, count, dtype, src, dst, stream) */
static PyObject* call_p2p(int which, PyObject* const* a, Py_ssize_t n) {
  void *comm, *buf, *stream;
  size_t count;
  int dtype, src, dst, rc;
  if (n_args(n, 7) || as_address(a[0], &comm) || as_address(a[1], &buf) || as_size(a[2], &count) || as_dtype(a[3], &dtype) ||
      as_int(a[4], &src) || as_int(a[5], &dst) || as_stream(a[6], &stream))
    return NULL;
  Py_BEGIN_ALLOW_THREADS
  rc = ((p2p_fn)g_fn[which])(buf, count, dtype, src, dst, comm, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

static PyObject* py_allreduce(PyObject* m, PyObject* const* a, Py_ssize_t n) { return call_with_op(F_ALLREDUCE, a, n); }
static PyObject* py_reduce_scatter(PyObject* m, PyObject* const* a, Py_ssize_t n) { return call_with_op(F_REDUCE_SCATTER, a, n); }
static PyObject* py_host_allreduce(PyObject* m, PyObject* const* a, Py_ssize_t n) { return call_with_op(F_HOST_ALLREDUCE, a, n); }
static PyObject* py_allgather(PyObject* m, PyObject* const* a, Py_ssize_t n) { return call_without_op(F_ALLGATHER, a, n); }
static PyObject* py_alltoall(PyObject* m, PyObject* const* a, Py_ssize_t n) { return call_without_op(F_ALLTOALL, a, n); }
static PyObject* py_send(PyObject* m, PyObject* const* a, Py_ssize_t n) { return call_p2p(F_SEND, a, n); }
static PyObject* py_recv(PyObject* m, PyObject* const* a, Py_ssize_t n) { return call_p2p(F_RECV, a, n); }

/* (send, recv, count, dtype, op, R, stream) */
static PyObject* py_allreduce_static(PyObject* m, PyObject* const* a, Py_ssize_t n) {
  void *send[MAX_RANKS], *recv[MAX_RANKS], *stream;
  size_t count;
  int dtype, op, R, rc;
  if (n_args(n, 7) || as_addresses(a[0], send) || as_addresses(a[1], recv) || as_size(a[2], &count) || as_dtype(a[3], &dtype) ||
      as_int(a[4], &op) || as_int(a[5], &R) || as_stream(a[6], &stream))
    return NULL;
  Py_BEGIN_ALLOW_THREADS
  rc = ((static_fn)g_fn[F_STATIC])((const void* const*)send, recv, count, dtype, op, R, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

/* R * R sizes */
static int as_sizes(PyObject* seq, size_t n, size_t* out) {
  PyObject* f = PySequence_Fast(seq, "a sequence of R * R numbers is wanted");
  if (!f) return -1;
  int rc = 0;
  const size_t given = (size_t)PySequence_Fast_GET_SIZE(f);
  if (given > n) {
    PyErr_Format(PyExc_IndexError, "%zu numbers, %zu wanted", given, n);
    rc = -1;
  }
  for (size_t i = 0; i < given && rc == 0; i++) rc = as_size(PySequence_Fast_GET_ITEM(f, (Py_ssize_t)i), &out[i]);
  for (size_t i = given; i < n; i++) out[i] = 0;
  Py_DECREF(f);
  return rc;
}

/* (comm, R, send, sendcounts, sdispls, recv, rdispls, dtype, stream) */
static PyObject* py_alltoallv(PyObject* m, PyObject* const* a, Py_ssize_t n) {
  void *send[MAX_RANKS], *recv[MAX_RANKS], *comm, *stream;
  int R, dtype, rc;
  if (n_args(n, 9) || as_address(a[0], &comm) || as_int(a[1], &R) || as_addresses(a[2], send) || as_addresses(a[5], recv) ||
      as_dtype(a[7], &dtype) || as_stream(a[8], &stream))
    return NULL;
  if (R < 1 || R > MAX_RANKS) {
    PyErr_SetString(PyExc_ValueError, "rank count out of range");
    return NULL;
  }
  const size_t k = (size_t)R * (size_t)R;
  size_t* buf = PyMem_Malloc(3 * k * sizeof(size_t));
  if (!buf) return PyErr_NoMemory();
  if (as_sizes(a[3], k, buf) || as_sizes(a[4], k, buf + k) || as_sizes(a[6], k, buf + 2 * k)) {
    PyMem_Free(buf);
    return NULL;
  }
  Py_BEGIN_ALLOW_THREADS
  rc = ((pattern_fn)g_fn[F_ALLTOALLV])((const void* const*)send, buf, buf + k, recv, buf + 2 * k, dtype, comm, stream);
  Py_END_ALLOW_THREADS
  PyMem_Free(buf);
  return PyLong_FromLong(rc);
}

/* The addresses of the library's functions, in the order of the enumeration above. */
static PyObject* py_bind(PyObject* m, PyObject* const* a, Py_ssize_t n) {
  if (n_args(n, F_COUNT)) return NULL;
  for (Py_ssize_t i = 0; i < n; i++)
    if (as_address(a[i], &g_fn[i])) return NULL;
  Py_RETURN_NONE;
}

#define ENTRY(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {ENTRY(bind),     ENTRY(allreduce), ENTRY(reduce_scatter), ENTRY(host_allreduce),
                                ENTRY(allgather), ENTRY(alltoall),  ENTRY(alltoallv),      ENTRY(send),
                                ENTRY(recv),      ENTRY(allreduce_static), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) {
  g_data_ptr = PyUnicode_InternFromString("data_ptr");
  g_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  return g_data_ptr && g_cuda_stream ? PyModule_Create(&module) : NULL;
}
