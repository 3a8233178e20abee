/*
 * Argument marshalling of the hot calls for Python: tensors to addresses, numbers to C types, one call of the library.
 * A request of 32 layers makes 64 of these calls, and a small request takes the GPU less time than ctypes took to issue it:
 * ba_final_attend 6.6 -> 4.0 us, ba_reencode_k 4.6 -> 2.8 us a call (a kernel launch included), a small request 33.4 -> 27.5 us.
 * Nothing else happens here; the functions are those of the library that bind() is given (the handle ctypes opened), their
 * prototypes the header's.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>
#include <stdint.h>

#include "ba.h"

static PyObject *s_data_ptr, *s_is_contiguous;

/* None -> NULL, an int -> that address, an object with data_ptr() (a contiguous torch tensor) -> its data, otherwise the
 * contiguous buffer of the object (numpy arrays, ctypes structures and handles). */
static int to_address(PyObject *o, void **out) {
  if (o == Py_None) { *out = NULL; return 1; }
  if (PyLong_Check(o)) {
    *out = PyLong_AsVoidPtr(o);
    return !(*out == NULL && PyErr_Occurred());
  }
  PyObject *r = PyObject_CallMethodNoArgs(o, s_is_contiguous);
  if (r) {
    const int yes = PyObject_IsTrue(r);
    Py_DECREF(r);
    if (yes < 0) return 0;
    if (!yes) { PyErr_SetString(PyExc_ValueError, "tensor must be contiguous"); return 0; }
    r = PyObject_CallMethodNoArgs(o, s_data_ptr);
    if (!r) return 0;
    *out = PyLong_AsVoidPtr(r);
    Py_DECREF(r);
    return !(*out == NULL && PyErr_Occurred());
  }
  if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return 0;
  PyErr_Clear();
  Py_buffer b;
  if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return 0;
  *out = b.buf;
  PyBuffer_Release(&b);
  return 1;
}
/* A ctypes structure or handle: the address of its memory. */
static int to_struct(PyObject *o, void **out) {
  Py_buffer b;
  if (o == Py_None) { *out = NULL; return 1; }
  if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return 0;
  *out = b.buf;
  PyBuffer_Release(&b);
  return 1;
}
static int to_context(PyObject *o, ba_ctx **out) {
  Py_buffer b;
  if (o == Py_None || PyLong_Check(o)) return to_address(o, (void **)out);
  if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return 0;
  *out = b.len == sizeof(void *) ? *(ba_ctx **)b.buf : NULL;
  PyBuffer_Release(&b);
  return 1;
}
static int to_int(PyObject *o, int32_t *out) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) return 0;
  if (v < INT32_MIN || v > INT32_MAX) { PyErr_SetString(PyExc_OverflowError, "argument does not fit 32 bits"); return 0; }
  *out = (int32_t)v;
  return 1;
}

#define ARGS(n) if (nargs != (n)) return PyErr_Format(PyExc_TypeError, "%d arguments expected, got %zd", (n), nargs)
#define P(i, v) void *v; if (!to_address(args[i], &v)) return NULL
#define I(i, v) int32_t v; if (!to_int(args[i], &v)) return NULL
#define CTX ba_ctx *ctx; if (!to_context(args[0], &ctx)) return NULL
#define S(i, v) void *v; if (!to_struct(args[i], &v)) return NULL
#define CALL(expr)                                   \
  do {                                               \
    ba_status st;                                    \
    Py_BEGIN_ALLOW_THREADS st = (expr);              \
    Py_END_ALLOW_THREADS return PyLong_FromLong(st); \
  } while (0)
#define FUNCTIONS(X) X(ba_segment) X(ba_reencode_k) X(ba_reencode_k_paged) X(ba_block_prefill) X(ba_block_prefill_bwd) \
  X(ba_final_attend) X(ba_final_attend_fused) X(ba_final_attend_paged) X(ba_final_attend_fused_paged)
#define DECLARE(f) static __typeof__(&f) p_##f;
FUNCTIONS(DECLARE)

static PyObject *m_segment(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(11); CTX; P(1, lens); P(2, nblocks); I(3, batch); I(4, n_blocks); I(5, n_tokens); I(6, mode); P(7, buf);
  const Py_ssize_t bytes = PyLong_AsSsize_t(args[8]);
  if (bytes == -1 && PyErr_Occurred()) return NULL;
  S(9, out); P(10, stream);
  CALL(p_ba_segment(ctx, lens, nblocks, batch, n_blocks, n_tokens, mode, buf, (size_t)bytes, out, stream));
}
static PyObject *m_reencode_k(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(10); CTX; P(1, src); P(2, off); I(3, n_src); P(4, dst); P(5, cu); P(6, delta); I(7, n_blocks); I(8, n_rows); P(9, stream);
  CALL(p_ba_reencode_k(ctx, src, off, n_src, dst, cu, delta, n_blocks, n_rows, stream));
}
static PyObject *m_reencode_k_paged(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(9); CTX; P(1, pool); S(2, pages); P(3, dst); P(4, cu); P(5, delta); I(6, n_blocks); I(7, n_rows); P(8, stream);
  CALL(p_ba_reencode_k_paged(ctx, pool, pages, dst, cu, delta, n_blocks, n_rows, stream));
}
static PyObject *m_block_prefill(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(10); CTX; P(1, q); P(2, k); P(3, v); P(4, o); P(5, lse); S(6, seg); I(7, mode); I(8, out); P(9, stream);
  CALL(p_ba_block_prefill(ctx, q, k, v, o, lse, seg, mode, out, stream));
}
static PyObject *m_block_prefill_bwd(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(14); CTX; P(1, q); P(2, k); P(3, v); P(4, o); P(5, lse); P(6, d_o); P(7, dq); P(8, dk); P(9, dv); S(10, seg); I(11, mode);
  I(12, out); P(13, stream);
  CALL(p_ba_block_prefill_bwd(ctx, q, k, v, o, lse, d_o, dq, dk, dv, seg, mode, out, stream));
}
static PyObject *m_final_attend(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(16); CTX; P(1, q); P(2, k); P(3, v); I(4, n_final); P(5, kc); P(6, vc); I(7, n_cache); P(8, voff); I(9, n_v); P(10, o);
  P(11, lse); S(12, seg); I(13, mode); I(14, out); P(15, stream);
  CALL(p_ba_final_attend(ctx, q, k, v, n_final, kc, vc, n_cache, voff, n_v, o, lse, seg, mode, out, stream));
}
static PyObject *m_final_attend_fused(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(17); CTX; P(1, q); P(2, k); P(3, v); I(4, n_final); P(5, ks); P(6, vs); I(7, n_src); P(8, off); I(9, n_cache); P(10, k_out);
  P(11, o); P(12, lse); S(13, seg); I(14, mode); I(15, out); P(16, stream);
  CALL(p_ba_final_attend_fused(ctx, q, k, v, n_final, ks, vs, n_src, off, n_cache, k_out, o, lse, seg, mode, out, stream));
}
static PyObject *m_final_attend_paged(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(15); CTX; P(1, q); P(2, k); P(3, v); I(4, n_final); P(5, kc); I(6, n_cache); P(7, pool); S(8, pages); P(9, o); P(10, lse);
  S(11, seg); I(12, mode); I(13, out); P(14, stream);
  CALL(p_ba_final_attend_paged(ctx, q, k, v, n_final, kc, n_cache, pool, pages, o, lse, seg, mode, out, stream));
}
static PyObject *m_final_attend_fused_paged(PyObject *self, PyObject *const *args, Py_ssize_t nargs) {
  ARGS(16); CTX; P(1, q); P(2, k); P(3, v); I(4, n_final); P(5, kp); P(6, vp); S(7, pages); I(8, n_cache); P(9, k_out); P(10, o);
  P(11, lse); S(12, seg); I(13, mode); I(14, out); P(15, stream);
  CALL(p_ba_final_attend_fused_paged(ctx, q, k, v, n_final, kp, vp, pages, n_cache, k_out, o, lse, seg, mode, out, stream));
}

/* bind(handle): take the library's functions from the shared object a dlopen handle names. */
static PyObject *m_bind(PyObject *self, PyObject *handle) {
  void *h = PyLong_AsVoidPtr(handle);
  if (!h && PyErr_Occurred()) return NULL;
#define RESOLVE(f) \
  if (!(p_##f = (__typeof__(&f))dlsym(h, #f))) return PyErr_Format(PyExc_RuntimeError, "%s is not in the library", #f);
  FUNCTIONS(RESOLVE)
  Py_RETURN_NONE;
}

#define METHOD(n) {#n, (PyCFunction)(void (*)(void))m_##n, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {{"bind", m_bind, METH_O, NULL}, METHOD(segment), METHOD(reencode_k), METHOD(reencode_k_paged),
                                METHOD(block_prefill), METHOD(block_prefill_bwd), METHOD(final_attend), METHOD(final_attend_fused),
                                METHOD(final_attend_paged), METHOD(final_attend_fused_paged), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "ba_marshal", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit_ba_marshal(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
  return s_data_ptr && s_is_contiguous ? PyModule_Create(&module) : NULL;
}
