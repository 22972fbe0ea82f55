// Argument marshalling of the Python entry points, as a CPython extension (_binding.<tag>.so).
//
// A call of a small problem is bound by the time its Python caller spends on it: building the descriptor field by field
// through ctypes, wrapping every pointer and asking for the current stream took 9 of the 13.5 us that a 16 x 256 x 64
// post-norm call cost the host (4.0 us of it inside the library).  This module reads the tensors' shapes, strides and
// addresses through their Python interface (no dependence on the tensor library's binary interface), fills the C structures
// and calls the entry point with the interpreter lock released.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "comfuse.h"

typedef comfuse_status_t (*gemm_epilogue_fn)(const comfuse_gemm_desc_t*, const void*, const void*, void*, const comfuse_epilogue_args_t*, void*, size_t, void*);
typedef comfuse_status_t (*b2b_gemm_fn)(const comfuse_b2b_desc_t*, const void*, const void*, const void*, const void*, const void*, const void*,
                                        const void*, void*, void*, size_t, void*);
typedef comfuse_status_t (*gemm_spec_fn)(const comfuse_fusion_spec_t*, const comfuse_gemm_shape_t*, const void*, const void*, void*, const void* const*,
                                         const int64_t*, void* const*, int32_t, void*, size_t, void*);
static gemm_epilogue_fn f_gemm_epilogue;
static b2b_gemm_fn f_b2b_gemm;
static gemm_spec_fn f_gemm_spec;
static PyObject *s_data_ptr, *s_shape, *s_stride, *s_dim, *s_is_contiguous, *s_numel, *s_element_size, *s_cuda_stream;

#define MAX_DIMS 64  // (tensors have no more)
typedef struct {
  int n;
  int64_t size[MAX_DIMS], stride[MAX_DIMS];
} Geometry;

static int to_i64(PyObject* o, int64_t* out) {  // int(o); wraps like a C integer
  PyObject* v = PyLong_Check(o) ? Py_NewRef(o) : PyNumber_Long(o);
  if (!v) return 0;
  *out = (int64_t)PyLong_AsUnsignedLongLongMask(v);
  Py_DECREF(v);
  return !PyErr_Occurred();
}
static int to_f64(PyObject* o, double* out) {  // float(o): numbers, tensors of one element, texts
  if (PyFloat_CheckExact(o)) {
    *out = PyFloat_AS_DOUBLE(o);
    return 1;
  }
  PyObject* v = PyNumber_Float(o);
  if (!v) return 0;
  *out = PyFloat_AS_DOUBLE(v);
  Py_DECREF(v);
  return 1;
}
static int tuple_i64(PyObject* t, int64_t* out, int* n) {
  PyObject* seq = t ? PySequence_Fast(t, "a shape or stride") : NULL;
  Py_XDECREF(t);
  if (!seq) return 0;
  const Py_ssize_t len = PySequence_Fast_GET_SIZE(seq);
  if (len > MAX_DIMS) {
    Py_DECREF(seq);
    PyErr_SetString(PyExc_AssertionError, "too many dimensions");
    return 0;
  }
  for (Py_ssize_t i = 0; i < len; ++i)
    if (!to_i64(PySequence_Fast_GET_ITEM(seq, i), out + i)) {
      Py_DECREF(seq);
      return 0;
    }
  *n = (int)len;
  Py_DECREF(seq);
  return 1;
}
static int shape_of(PyObject* t, Geometry* g) { return tuple_i64(PyObject_GetAttr(t, s_shape), g->size, &g->n); }
static int geometry(PyObject* t, Geometry* g) {
  int n = 0;
  if (!shape_of(t, g) || !tuple_i64(PyObject_CallMethodNoArgs(t, s_stride), g->stride, &n)) return 0;
  if (n != g->n || n < 2) {
    PyErr_SetString(PyExc_IndexError, "Dimension out of range (a matrix or a batch of matrices is expected)");
    return 0;
  }
  return 1;
}
static int method_i64(PyObject* t, PyObject* name, int64_t* out) {
  PyObject* v = PyObject_CallMethodNoArgs(t, name);
  if (!v) return 0;
  const int ok = to_i64(v, out);
  Py_DECREF(v);
  return ok;
}
static int pointer(PyObject* t, const void** out) {  // None: a null pointer
  int64_t v = 0;
  if (t != Py_None && !method_i64(t, s_data_ptr, &v)) return 0;
  *out = (const void*)(uintptr_t)v;
  return 1;
}
static int workspace_of(PyObject* t, void** ptr, size_t* bytes) {
  int64_t n = 0, size = 0;
  *bytes = 0;
  if (!pointer(t, (const void**)ptr)) return 0;
  if (t == Py_None) return 1;
  if (!method_i64(t, s_numel, &n) || !method_i64(t, s_element_size, &size)) return 0;
  *bytes = (size_t)(n * size);
  return 1;
}
static int contiguous(PyObject* t) {
  PyObject* v = PyObject_CallMethodNoArgs(t, s_is_contiguous);
  if (!v) return 0;
  const int yes = PyObject_IsTrue(v);
  Py_DECREF(v);
  if (yes == 0) PyErr_SetString(PyExc_AssertionError, "a dense tensor is expected");
  return yes == 1;
}
static int require(int cond, const char* what) {
  if (!cond) PyErr_SetString(PyExc_AssertionError, what);
  return cond;
}
// a stream object (which may be callable), or the function that returns the current stream's handle
static int stream_of(PyObject* s, void** out) {
  PyObject* v = PyFunction_Check(s) ? PyObject_CallNoArgs(s) : PyObject_GetAttr(s, s_cuda_stream);
  int64_t h = 0;
  if (!v) return 0;
  const int ok = to_i64(v, &h);
  Py_DECREF(v);
  *out = (void*)(uintptr_t)h;
  return ok;
}
static int fixed_args(Py_ssize_t got, Py_ssize_t want, const char* name) {
  if (got != want) PyErr_Format(PyExc_TypeError, "%s takes %zd arguments, got %zd", name, want, got);
  return got == want;
}

// a = (A, B, Y, kind, residual, alpha, eps, mask, fused, flags, softcap)
static int fill_desc(PyObject* const* a, comfuse_gemm_desc_t* d) {
  Geometry A, B, Y, R;
  int64_t kind, mask, flags;
  if (!geometry(a[0], &A) || !geometry(a[1], &B) || !geometry(a[2], &Y)) return 0;
  if (!to_i64(a[9], &flags)) return 0;
  const int batched = A.n == 3, b_nk = (flags & COMFUSE_FLAG_B_ROW_MAJOR_NK) != 0;
  const int64_t M = A.size[A.n - 2], K = A.size[A.n - 1], N = B.size[B.n - (b_nk ? 2 : 1)];
  if (!require(B.size[B.n - (b_nk ? 1 : 2)] == K && Y.size[Y.n - 2] == M && Y.size[Y.n - 1] == N, "shapes of A, B and Y do not match")) return 0;
  if (!require(A.stride[A.n - 1] == 1 && B.stride[B.n - 1] == 1 && Y.stride[Y.n - 1] == 1, "the last dimension of A, B and Y must be dense")) return 0;
  memset(d, 0, sizeof(*d));
  d->batch = (int32_t)(batched ? A.size[0] : 1);
  d->M = (int32_t)M;
  d->N = (int32_t)N;
  d->K = (int32_t)K;
  d->lda = A.stride[A.n - 2];
  d->ldb = B.stride[B.n - 2];
  d->ldy = Y.stride[Y.n - 2];
  d->batch_stride_a = batched ? A.stride[0] : M * d->lda;
  d->batch_stride_b = batched ? B.stride[0] : (b_nk ? N : K) * d->ldb;
  d->batch_stride_y = batched ? Y.stride[0] : M * d->ldy;
  d->ldr = N;
  d->batch_stride_r = M * N;
  if (a[4] != Py_None) {
    if (!geometry(a[4], &R)) return 0;
    d->ldr = R.stride[R.n - 2];
    d->batch_stride_r = batched ? R.stride[0] : M * d->ldr;
  }
  if (!to_i64(a[3], &kind) || !to_i64(a[7], &mask)) return 0;
  double alpha, eps, softcap;
  if (!to_f64(a[5], &alpha) || !to_f64(a[6], &eps) || !to_f64(a[10], &softcap)) return 0;
  const int fused = PyObject_IsTrue(a[8]);
  if (fused < 0) return 0;
  d->kind = (int32_t)kind;
  d->mask = (int32_t)mask;
  d->alpha = (float)alpha;
  d->eps = (float)eps;
  d->fused = fused;
  d->flags = (uint32_t)flags;
  d->softcap = (float)softcap;
  return 1;
}

// gemm_desc(A, B, Y, kind, residual, alpha, eps, mask, fused, flags, softcap) -> bytes of a comfuse_gemm_desc_t
static PyObject* py_gemm_desc(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  comfuse_gemm_desc_t d;
  if (!fixed_args(n, 11, "gemm_desc") || !fill_desc(a, &d)) return NULL;
  return PyBytes_FromStringAndSize((const char*)&d, sizeof(d));
}

// gemm_epilogue(<the arguments of gemm_desc>, bias, gamma, beta, mask_tensor, row_max, row_argmax, workspace, stream) -> status
static PyObject* py_gemm_epilogue(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  comfuse_gemm_desc_t d;
  comfuse_epilogue_args_t e;
  const void *A, *B, *Y;
  void *ws, *stream;
  size_t ws_bytes;
  if (!fixed_args(n, 19, "gemm_epilogue") || !fill_desc(a, &d)) return NULL;
  memset(&e, 0, sizeof(e));
  if (!pointer(a[11], &e.bias) || !pointer(a[4], &e.residual) || !pointer(a[12], &e.gamma) || !pointer(a[13], &e.beta) || !pointer(a[14], &e.mask) ||
      !pointer(a[15], (const void**)&e.row_max) || !pointer(a[16], (const void**)&e.row_argmax) || !workspace_of(a[17], &ws, &ws_bytes) ||
      !pointer(a[0], &A) || !pointer(a[1], &B) || !pointer(a[2], &Y) || !stream_of(a[18], &stream))
    return NULL;
  comfuse_status_t st;
  Py_BEGIN_ALLOW_THREADS
  st = f_gemm_epilogue(&d, A, B, (void*)Y, &e, ws, ws_bytes, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong((long)st);
}

// b2b(kind, X, W1, b1, W2, b2, gamma, beta, O, eps, alpha, fused, flags, workspace, stream) -> status
static PyObject* py_b2b(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  comfuse_b2b_desc_t d;
  Geometry X, W1, W2, O;
  int64_t kind, flags;
  if (!fixed_args(n, 15, "b2b") || !to_i64(a[0], &kind) || !to_i64(a[12], &flags)) return NULL;
  const int attention = kind == COMFUSE_B2B_SOFTMAX_ATTENTION;
  if (!shape_of(a[1], &X) || !shape_of(a[2], &W1) || !shape_of(a[4], &W2)) return NULL;
  if (X.n != (attention ? 3 : 2)) {
    PyErr_Format(PyExc_ValueError, "a tensor of %d dimensions is expected, got %d", attention ? 3 : 2, X.n);
    return NULL;
  }
  if (W2.n <= (attention ? 2 : 1) || (!attention && W1.n < 2)) {
    PyErr_SetString(PyExc_IndexError, "tuple index out of range");
    return NULL;
  }
  memset(&d, 0, sizeof(d));
  const int64_t nb = attention ? X.size[0] : 1, M = X.size[X.n - 2], K = X.size[X.n - 1];
  const int64_t N1 = attention ? W2.size[1] : W1.size[1], N2 = attention ? W2.size[2] : W2.size[1];
  if (attention) {
    const int rm = (flags & COMFUSE_B2B_FLAG_KEYS_ROW_MAJOR) != 0;
    if (!shape_of(a[8], &O)) return NULL;
    if (!require(W1.n == 3 && W1.size[0] == nb && W1.size[1] == (rm ? N1 : K) && W1.size[2] == (rm ? K : N1) && W2.n == 3 && W2.size[0] == nb && O.n == 3 &&
                     O.size[0] == nb && O.size[1] == M && O.size[2] == N2,
                 "shapes of Q, keys, V and O do not match"))
      return NULL;
  } else if (kind == COMFUSE_B2B_MLP_RELU) {
    if (!shape_of(a[8], &O)) return NULL;
    if (!require(W1.n == 2 && W1.size[0] == K && W2.n == 2 && W2.size[0] == N1 && O.n == 2 && O.size[0] == M && O.size[1] == N2, "shapes of X, W1, W2 and O do not match"))
      return NULL;
  }
  if (!contiguous(a[1]) || !contiguous(a[2]) || !contiguous(a[4]) || !contiguous(a[8])) return NULL;
  double eps, alpha;
  if (!to_f64(a[9], &eps) || !to_f64(a[10], &alpha)) return NULL;
  const int fused = PyObject_IsTrue(a[11]);
  if (fused < 0) return NULL;
  d.M = (int32_t)M;
  d.K = (int32_t)K;
  d.N1 = (int32_t)N1;
  d.N2 = (int32_t)N2;
  d.eps = (float)eps;
  d.fused = fused;
  d.kind = (int32_t)kind;
  d.batch = (int32_t)nb;
  d.alpha = (float)alpha;
  d.flags = (int32_t)flags;
  const void* p[8];
  void *ws, *stream;
  size_t ws_bytes;
  for (int i = 0; i < 8; ++i)
    if (!pointer(a[1 + i], p + i)) return NULL;
  if (!workspace_of(a[13], &ws, &ws_bytes) || !stream_of(a[14], &stream)) return NULL;
  comfuse_status_t st;
  Py_BEGIN_ALLOW_THREADS
  st = f_b2b_gemm(&d, p[0], p[1], p[2], p[3], p[4], p[5], p[6], (void*)p[7], ws, ws_bytes, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong((long)st);
}

// A sequence of tensors (something with a length: a generator's tensors would be gone before the launch is enqueued), held for the
// length of a call, and zeroed room for `arrays` 8-byte values of each.  The library reads as many entries as the program
// names, so there is room for the most that a program can name, however few were given.
#define MIN_ROOM (COMFUSE_SPEC_MAX_PARAMS > COMFUSE_SPEC_MAX_ROW_OUTPUTS ? COMFUSE_SPEC_MAX_PARAMS : COMFUSE_SPEC_MAX_ROW_OUTPUTS)
typedef struct {
  PyObject* seq;
  Py_ssize_t n, room;
  int64_t* values;
} Held;
static int hold(PyObject* o, int arrays, Held* h) {
  if (PyObject_Size(o) < 0) return 0;
  h->seq = PySequence_Fast(o, "a sequence of tensors is expected");
  if (!h->seq) return 0;
  h->n = PySequence_Fast_GET_SIZE(h->seq);
  h->room = h->n > MIN_ROOM ? h->n : MIN_ROOM;
  h->values = PyMem_Calloc((size_t)(h->room * arrays), sizeof(int64_t));
  if (!h->values) PyErr_NoMemory();
  return h->values != NULL;
}
static void let_go(Held* h) {
  PyMem_Free(h->values);
  Py_XDECREF(h->seq);
}

// gemm_spec(A, B, Y, address of the comfuse_fusion_spec_t, params, row_out, fused, b_nk, workspace, stream) -> status
static int gemm_spec_call(PyObject* const* a, Held* params, Held* rows, comfuse_status_t* st) {
  Geometry A, B, Y;
  comfuse_gemm_shape_t s;
  int64_t spec, fused;
  if (!geometry(a[0], &A) || !geometry(a[1], &B) || !geometry(a[2], &Y) || !to_i64(a[3], &spec) || !to_i64(a[6], &fused)) return 0;
  const int b_nk = PyObject_IsTrue(a[7]);
  if (b_nk < 0) return 0;
  const int batched = A.n == 3;
  memset(&s, 0, sizeof(s));
  const int64_t M = A.size[A.n - 2], K = A.size[A.n - 1], N = B.size[B.n - (b_nk ? 2 : 1)];
  s.batch = (int32_t)(batched ? A.size[0] : 1);
  s.M = (int32_t)M;
  s.N = (int32_t)N;
  s.K = (int32_t)K;
  s.lda = A.stride[A.n - 2] ? A.stride[A.n - 2] : K;
  s.ldb = B.stride[B.n - 2] ? B.stride[B.n - 2] : (b_nk ? K : N);
  s.ldy = Y.stride[Y.n - 2] ? Y.stride[Y.n - 2] : N;
  s.batch_stride_a = batched && A.stride[0] ? A.stride[0] : M * s.lda;
  s.batch_stride_b = batched && B.stride[0] ? B.stride[0] : (b_nk ? N : K) * s.ldb;
  s.batch_stride_y = batched && Y.stride[0] ? Y.stride[0] : M * s.ldy;
  s.flags = b_nk ? COMFUSE_FLAG_B_ROW_MAJOR_NK : 0;
  if (!hold(a[4], 2, params) || !hold(a[5], 1, rows)) return 0;
  int64_t* ld = params->values + params->room;
  for (Py_ssize_t i = 0; i < params->n; ++i) {
    PyObject* t = PySequence_Fast_GET_ITEM(params->seq, i);
    int64_t dims = 0;
    Geometry g;
    if (t == Py_None) continue;
    if (!method_i64(t, s_data_ptr, params->values + i) || !method_i64(t, s_dim, &dims)) return 0;
    if (dims < 2) continue;
    if (!geometry(t, &g)) return 0;
    ld[i] = g.stride[g.n - 2];
  }
  for (Py_ssize_t i = 0; i < rows->n; ++i)
    if (!method_i64(PySequence_Fast_GET_ITEM(rows->seq, i), s_data_ptr, rows->values + i)) return 0;
  const void *pA, *pB, *pY;
  void *ws, *stream;
  size_t ws_bytes;
  if (!workspace_of(a[8], &ws, &ws_bytes) || !pointer(a[0], &pA) || !pointer(a[1], &pB) || !pointer(a[2], &pY) || !stream_of(a[9], &stream)) return 0;
  Py_BEGIN_ALLOW_THREADS
  *st = f_gemm_spec((const comfuse_fusion_spec_t*)(uintptr_t)spec, &s, pA, pB, (void*)pY, (const void* const*)params->values, ld, (void* const*)rows->values,
                    (int32_t)fused, ws, ws_bytes, stream);
  Py_END_ALLOW_THREADS
  return 1;
}
static PyObject* py_gemm_spec(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Held params = {0}, rows = {0};
  comfuse_status_t st;
  if (!fixed_args(n, 10, "gemm_spec")) return NULL;
  const int ok = gemm_spec_call(a, &params, &rows, &st);
  let_go(&params);
  let_go(&rows);
  return ok ? PyLong_FromLong((long)st) : NULL;
}

// bind(address of comfuse_gemm_epilogue, of comfuse_b2b_gemm, of comfuse_gemm_spec): the loaded library's entry points
static PyObject* py_bind(PyObject* self, PyObject* args) {
  unsigned long long e, b, s;
  if (!PyArg_ParseTuple(args, "KKK", &e, &b, &s)) return NULL;
  f_gemm_epilogue = (gemm_epilogue_fn)(uintptr_t)e;
  f_b2b_gemm = (b2b_gemm_fn)(uintptr_t)b;
  f_gemm_spec = (gemm_spec_fn)(uintptr_t)s;
  Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"bind", py_bind, METH_VARARGS, NULL},
    {"gemm_desc", (PyCFunction)(void (*)(void))py_gemm_desc, METH_FASTCALL, NULL},
    {"gemm_epilogue", (PyCFunction)(void (*)(void))py_gemm_epilogue, METH_FASTCALL, NULL},
    {"b2b", (PyCFunction)(void (*)(void))py_b2b, METH_FASTCALL, NULL},
    {"gemm_spec", (PyCFunction)(void (*)(void))py_gemm_spec, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_binding", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__binding(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_shape = PyUnicode_InternFromString("shape");
  s_stride = PyUnicode_InternFromString("stride");
  s_dim = PyUnicode_InternFromString("dim");
  s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
  s_numel = PyUnicode_InternFromString("numel");
  s_element_size = PyUnicode_InternFromString("element_size");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  return PyModule_Create(&module);
}
